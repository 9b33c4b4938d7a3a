// Thin inline-PTX layer for sm_100a: mbarriers with bounded waits, TMA tile copies,
// tensor memory (TMEM) management, tcgen05 MMA issue / commit / load / store, and the
// shared-memory matrix descriptors and instruction descriptor the MMA consumes.
//
// Nothing here knows about attention; the kernels in this directory build on it.
#pragma once

#include <cstdint>
#include <cuda.h>          // CUtensorMap (types only; the driver entry point is fetched at run time)
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace moda {

// ------------------------------------------------------------------------------------
// Device status word.  A bounded wait that runs out records where it gave up here; the
// host reads it with moda_last_status().  0 = no error.
// ------------------------------------------------------------------------------------
__device__ int g_moda_status = 0;
// Mirror of the status word in host memory that the device can write (set up by the host on its first
// call on a device; null until then).  Written only when a wait runs out, so that the next host call
// can see the failure with a plain load instead of a device synchronisation.
__device__ int* g_moda_status_host = nullptr;

enum : int {
    kStatusOk = 0,
    kStatusWaitTimeout = 1,   // | (site << 8)
    kStatusSmemLayout = 2,    // the dynamic shared-memory segment is too small for the kernel's plan
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 1024-aligned start of the dynamic shared-memory segment, or nullptr if `need` bytes do not fit
// behind it (reported through the status word by the caller).
__device__ __forceinline__ uint8_t* aligned_dynamic_smem(uint8_t* raw, uint32_t need) {
    uint8_t* p = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    uint32_t dyn;
    asm volatile("mov.u32 %0, %dynamic_smem_size;" : "=r"(dyn));
    return (uint32_t(p - raw) + need <= dyn) ? p : nullptr;
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "elect.sync _|p, 0xffffffff;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(pred));
    return pred != 0;
}

// Programmatic dependent launch.  The first lets the next grid of the stream start (if it was launched to) once every CTA
// of this one has said so or ended; the second returns when the grids that this one was launched beside have ended and
// their writes are visible.
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Warpgroup-wide register re-allocation (all 128 threads of the warpgroup execute it).
template <int N>
__device__ __forceinline__ void setmaxnreg_inc() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void setmaxnreg_dec() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

// ------------------------------------------------------------------------------------
// mbarrier
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait.  `abort_flag` is a CTA-wide word in shared memory: the first wait that runs out leaves its site's code there,
// and from then on every wait of the CTA gives up after two probes so that the CTA can reach its tear-down (TMEM release)
// instead of spinning; there abort_teardown passes the code on.  Limit: 2e9 cycles, about 1 s (the cycle counter: a read of
// the global timer takes about a microsecond, which every wait that has to wait would pay).
//
// What a wait site costs in code matters: a kernel here has ten to thirty of them in its loops.  With the clock in 64
// bits, a spin counter and the report in line (some 45 instructions a site), and the loops around them unrolled by the
// compiler, the kernels were 63 to 94 KB, the code that all warp roles run per iteration no longer fitted the
// instruction cache of an SM: the fused backward missed it on every fifth request, and its warps stood for a tenth of their
// time without an instruction to issue (smsp__average_warps_issue_stalled_no_instruction 1.28 of 12.2 per issue at T = 8192,
// l = 0; now 0.27 of 12.4).  So: one asm block whose usual path is a few instructions, loops over tiles marked `unroll 1`,
// and code that few iterations need kept off their path.
// (32 probes without the clock before the bounded loop: 0-4 % slower forwards at d = 64 than this shorter form.)
__device__ __forceinline__ void report_abort(int code) {
    if (atomicCAS(&g_moda_status, 0, code) == 0) {
        int* host = g_moda_status_host;
        if (host != nullptr) {
            *reinterpret_cast<volatile int*>(host) = code;
            __threadfence_system();
        }
    }
}
// Every kernel that waits with mbar_wait calls this at its end, all threads, behind a CTA-wide barrier; another CTA-wide
// barrier follows, so that no thread leaves before the one that is named here.  If a wait gave up, that thread reports it
// and gives bulk copies still in flight a bounded time to land before the CTA's shared memory is handed on.  (The thread
// index is read again: kept over the kernel's loops it cost bwd_rows_kernel a register and 1-2 % with an e4m3 cache.)
__device__ __forceinline__ void abort_teardown(volatile int* abort_flag, uint32_t thread) {
    uint32_t tid;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
    if (*abort_flag != 0 && tid == thread) {
        report_abort(*abort_flag);
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 2000000ull) {}
    }
}
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int site,
                                          uint32_t limit_cycles = 2000000000u) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        ".reg .b32 t0, t;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%0], %1;\n"
        "@p bra DONE_%=;\n"
        "mov.u32 t0, %%clock;\n"
        "LONG_%=:\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%0], %1;\n"
        "@p bra DONE_%=;\n"
        "ld.volatile.shared.b32 t, [%2];\n"
        "setp.ne.b32 p, t, 0;\n"
        "@p bra DONE_%=;\n"
        "mov.u32 t, %%clock;\n"
        "sub.u32 t, t, t0;\n"
        "setp.lt.u32 p, t, %4;\n"
        "@p bra LONG_%=;\n"
        "atom.shared.cas.b32 t, [%2], 0, %3;\n"
        "DONE_%=:\n"
        "}\n"
        ::"r"(bar), "r"(parity), "r"(smem_u32(const_cast<const int*>(abort_flag))), "r"(kStatusWaitTimeout | (site << 8)), "r"(limit_cycles)
        : "memory");
}

// Bounded wait on two barriers.  Both probes are issued before either result is used, so their
// round trips through the shared-memory pipe (100-200 cycles each even when the phase is long
// complete) overlap; whatever is still pending afterwards is waited for one by one.
__device__ __forceinline__ void mbar_wait2(uint32_t bar_a, uint32_t parity_a, uint32_t bar_b, uint32_t parity_b,
                                           volatile int* abort_flag, int site_a, int site_b) {
    uint32_t ok_a, ok_b;
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%2], %3;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 q, [%4], %5;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "selp.u32 %1, 1, 0, q;\n"
        "}\n"
        : "=r"(ok_a), "=r"(ok_b)
        : "r"(bar_a), "r"(parity_a), "r"(bar_b), "r"(parity_b)
        : "memory");
    if (!ok_a) mbar_wait(bar_a, parity_a, abort_flag, site_a);
    if (!ok_b) mbar_wait(bar_b, parity_b, abort_flag, site_b);
}

// ------------------------------------------------------------------------------------
// Proxy / tcgen05 fences
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after_sync() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// ------------------------------------------------------------------------------------
// TMA (tiled bulk tensor copies).  The innermost coordinate times the element size must
// be a multiple of 16 bytes; all call sites use multiples of 64 bf16 elements.
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t smem_dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* m, uint32_t smem_src,
                                             int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
        ::"l"(reinterpret_cast<uint64_t>(m)), "r"(smem_src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
__device__ __forceinline__ void tma_store_commit() {
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void tma_store_wait_all() {
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}
// The same up to the point where the sources have been read: what a CTA needs before it gives its shared memory up (the
// writes belong to the grid, which ends after them).
__device__ __forceinline__ void tma_store_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// Plain (untiled) bulk copy global -> shared; both addresses 16-byte aligned, size a multiple
// of 16 bytes.  `policy` is an L2 cache policy made by l2_policy_evict_first().
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void bulk_load(uint32_t smem_dst, const void* gsrc, uint32_t bytes, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
        ::"r"(smem_dst), "l"(reinterpret_cast<uint64_t>(gsrc)), "r"(bytes), "r"(bar), "l"(policy)
        : "memory");
}

// ------------------------------------------------------------------------------------
// Tensor memory
// ------------------------------------------------------------------------------------
// One full warp allocates `ncols` (power of two, 32..512) columns; the base address is
// written to the shared-memory word at `smem_result`.
__device__ __forceinline__ void tmem_alloc(uint32_t smem_result, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// ------------------------------------------------------------------------------------
// CTA pairs (cta_group::2): two CTAs of a cluster whose tensor cores work on one 256-row tile.  Each CTA holds its own
// 128 rows of A, half of B's rows and its 128 lanes of the accumulator; the even CTA of the pair issues.
// ------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_cta_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// The address, in the cluster's shared-memory window, of the word that CTA `rank` has at this CTA's `addr`.
__device__ __forceinline__ uint32_t cluster_map_shared(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// Every thread of both CTAs; orders the mbarrier initialisation and shared-memory accesses across the pair.
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// TMA load whose completion bytes go to an mbarrier of the pair's other CTA (`bar` is a cluster-window address).
__device__ __forceinline__ void tma_load_4d_pair(uint32_t smem_dst, const CUtensorMap* m, uint32_t bar,
                                                 int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
// The same warp index of both CTAs calls these together.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_result, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// ------------------------------------------------------------------------------------
// Descriptors
// ------------------------------------------------------------------------------------
// 32-bit instruction descriptor for kind::f16 with bf16 operands and an fp32 accumulator.
//   [4,6) D format (1 = f32)   [7,10) A format (1 = bf16)   [10,13) B format (1 = bf16)
//   [15] A is MN-major         [16] B is MN-major
//   [17,23) N >> 3             [24,29) M >> 4
__host__ __device__ constexpr uint32_t make_idesc_bf16(int M, int N, bool a_mn_major, bool b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(a_mn_major) << 15) | (uint32_t(b_mn_major) << 16) |
           (uint32_t(N >> 3) << 17) | (uint32_t(M >> 4) << 24);
}

// 64-bit shared-memory matrix descriptor, 128-byte swizzle.
//   [0,14) start address >> 4      [16,30) leading-dimension byte offset >> 4
//   [32,46) stride-dimension byte offset >> 4      [46,48) version = 1      [61,64) layout = 2 (128B swizzle)
__device__ __forceinline__ uint64_t make_smem_desc_sw128(uint32_t smem_addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    uint64_t d = 0;
    d |= uint64_t((smem_addr & 0x3ffffu) >> 4);
    d |= uint64_t((lbo_bytes >> 4) & 0x3fffu) << 16;
    d |= uint64_t((sbo_bytes >> 4) & 0x3fffu) << 32;
    d |= uint64_t(1) << 46;
    d |= uint64_t(2) << 61;
    return d;
}

// Unswizzled K-major operand: core matrices of 8 rows x 16 bytes stored contiguously (128 bytes); `sbo_bytes` from one
// 8-row group to the next (M / N direction), `lbo_bytes` from the first 8 contraction elements to the second 8.
__device__ __forceinline__ uint64_t make_smem_desc_noswz(uint32_t smem_addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    uint64_t d = 0;
    d |= uint64_t((smem_addr & 0x3ffffu) >> 4);
    d |= uint64_t((lbo_bytes >> 4) & 0x3fffu) << 16;
    d |= uint64_t((sbo_bytes >> 4) & 0x3fffu) << 32;
    d |= uint64_t(1) << 46;
    return d;
}

// A tile stored as [rows][64 bf16] (128-byte rows, 8-row swizzle atoms of 1024 bytes), as a
// TMA box {64, rows} with 128B swizzle leaves it.
//  * used K-major (the 64-wide direction is the contraction): rows are M/N; successive 8-row
//    groups are 1024 bytes apart (stride offset); K advances by 32 bytes per 16 elements.
__device__ __forceinline__ uint64_t desc_kmajor_sw128(uint32_t tile_addr, int k16_step) {
    return make_smem_desc_sw128(tile_addr + uint32_t(k16_step) * 32u, 16u, 1024u);
}
//  * used MN-major (the rows are the contraction, the 64-wide direction is M/N): successive
//    8-row K groups are 1024 bytes apart (stride offset); the next 64 M/N elements live in the
//    next sub-tile, `mn_atom_bytes` further (leading offset); K advances by 16 rows = 2048 bytes.
__device__ __forceinline__ uint64_t desc_mnmajor_sw128(uint32_t tile_addr, int k16_step, uint32_t mn_atom_bytes) {
    return make_smem_desc_sw128(tile_addr + uint32_t(k16_step) * 2048u, mn_atom_bytes, 1024u);
}

// ------------------------------------------------------------------------------------
// tcgen05 MMA (issued by ONE thread), commit, load, store
// ------------------------------------------------------------------------------------
// The MMA-issuing code is run by a whole warp with warp-uniform operands and one elected lane
// issuing each instruction: the descriptors then live in uniform registers, which roughly halves
// what one tcgen05.mma costs its issuer compared with a loop that only lane 0 enters.
// D[tmem] (+)= A[smem] * B[smem]^T
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "elect.sync _|q, 0xffffffff;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]^T   (A: M rows on the lanes, K packed two bf16 per column)
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "elect.sync _|q, 0xffffffff;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
        "}\n"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// D[tmem of both CTAs] (+)= A[256 rows: 128 in each CTA's shared memory] * B[N rows: N / 2 in each CTA's]^T; issued
// by the pair's even CTA with descriptors that hold for both CTAs (same offsets).
__device__ __forceinline__ void umma_ss_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "elect.sync _|q, 0xffffffff;\n"
        "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive on `bar` (a cluster-window address: either CTA's barrier) once the pair MMAs issued so far have completed.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "elect.sync _|q, 0xffffffff;\n"
        "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
        "}\n" ::"r"(bar) : "memory");
}
// Arrive on `bar` once every MMA issued so far by this warp has completed (whole warp calls it, the
// elected lane -- the same lane that issued the MMAs -- executes it).
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "elect.sync _|q, 0xffffffff;\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
        "}\n" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Warp-collective: lane i of the warp reads TMEM lane (lane field of taddr + i), 32 / 16
// consecutive 32-bit columns starting at the column field of taddr.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr),
          "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr),
          "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
// 8 columns from r[off .. off + 7] (off a compile-time constant after unrolling).
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
        : "memory");
}

// ------------------------------------------------------------------------------------
// Small numeric helpers
// ------------------------------------------------------------------------------------
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Three-input maximum (one instruction; plain max.f32 issues at half rate on sm_100).
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// Two floats -> packed bf16x2 (lo in the low 16 bits), round to nearest even.
// Adds packed bf16 pairs to global memory (the adds happen in L2; nothing is returned).
__device__ __forceinline__ void red_add_bf16x2_v4(void* gptr, const uint4& v) {
    asm volatile("red.global.add.noftz.v4.bf16x2 [%0], {%1, %2, %3, %4};"
                 :: "l"(gptr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void red_add_f32_v4(float* gptr, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" :: "l"(gptr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
__device__ __forceinline__ void red_add_bf16x2_v2(void* gptr, const uint2& v) {
    asm volatile("red.global.add.noftz.v2.bf16x2 [%0], {%1, %2};" :: "l"(gptr), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void red_add_bf16x2(void* gptr, uint32_t v) {
    asm volatile("red.global.add.noftz.bf16x2 [%0], %1;" :: "l"(gptr), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// acc + lo(a) lo(b) + hi(a) hi(b), in this order: two mixed-precision FMAs (bf16 factors, fp32 sum), each rounded once like
// fmaf on the unpacked values, without the four instructions that unpack them.
__device__ __forceinline__ float fma_bf16x2(uint32_t a, uint32_t b, float acc) {
    asm("{\n"
        ".reg .b16 al, ah, bl, bh;\n"
        "mov.b32 {al, ah}, %1;\n"
        "mov.b32 {bl, bh}, %2;\n"
        "fma.rn.f32.bf16 %0, al, bl, %0;\n"
        "fma.rn.f32.bf16 %0, ah, bh, %0;\n"
        "}\n" : "+f"(acc) : "r"(a), "r"(b));
    return acc;
}
// The same into two sums: acc_lo + lo(a) lo(b), acc_hi + hi(a) hi(b).
__device__ __forceinline__ void fma2_bf16x2(uint32_t a, uint32_t b, float& acc_lo, float& acc_hi) {
    asm("{\n"
        ".reg .b16 al, ah, bl, bh;\n"
        "mov.b32 {al, ah}, %2;\n"
        "mov.b32 {bl, bh}, %3;\n"
        "fma.rn.f32.bf16 %0, al, bl, %0;\n"
        "fma.rn.f32.bf16 %1, ah, bh, %1;\n"
        "}\n" : "+f"(acc_lo), "+f"(acc_hi) : "r"(a), "r"(b));
}
// (y0, y1) += a * (lo(x), hi(x)): one packed fp32 FMA, each half rounded like fmaf.
__device__ __forceinline__ void axpy_bf16x2(float a, uint32_t x, float& y0, float& y1) {
    const uint32_t lo = x << 16, hi = x & 0xffff0000u;
    asm("{\n"
        ".reg .b64 aa, xx, yy;\n"
        "mov.b64 aa, {%2, %2};\n"
        "mov.b64 xx, {%3, %4};\n"
        "mov.b64 yy, {%0, %1};\n"
        "fma.rn.f32x2 yy, aa, xx, yy;\n"
        "mov.b64 {%0, %1}, yy;\n"
        "}\n" : "+f"(y0), "+f"(y1) : "f"(a), "r"(lo), "r"(hi));
}
// (y0, y1) += (a0, a1) * (b0, b1): one packed fp32 FMA, each half rounded like fmaf.
__device__ __forceinline__ void fma2_f32(float a0, float a1, float b0, float b1, float& y0, float& y1) {
    asm("{\n"
        ".reg .b64 aa, bb, yy;\n"
        "mov.b64 aa, {%2, %3};\n"
        "mov.b64 bb, {%4, %5};\n"
        "mov.b64 yy, {%0, %1};\n"
        "fma.rn.f32x2 yy, aa, bb, yy;\n"
        "mov.b64 {%0, %1}, yy;\n"
        "}\n" : "+f"(y0), "+f"(y1) : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}
// (y0, y1) = (x0, x1) * a + c and (x0 * z0, x1 * z1): packed fp32, each half rounded like fmaf / a product.
__device__ __forceinline__ void fma2_scale(float x0, float x1, float a, float c, float& y0, float& y1) {
    asm("{\n"
        ".reg .b64 xx, aa, cc;\n"
        "mov.b64 xx, {%2, %3};\n"
        "mov.b64 aa, {%4, %4};\n"
        "mov.b64 cc, {%5, %5};\n"
        "fma.rn.f32x2 xx, xx, aa, cc;\n"
        "mov.b64 {%0, %1}, xx;\n"
        "}\n" : "=f"(y0), "=f"(y1) : "f"(x0), "f"(x1), "f"(a), "f"(c));
}
__device__ __forceinline__ void mul2_f32(float x0, float x1, float z0, float z1, float& y0, float& y1) {
    asm("{\n"
        ".reg .b64 xx, zz;\n"
        "mov.b64 xx, {%2, %3};\n"
        "mov.b64 zz, {%4, %5};\n"
        "mul.rn.f32x2 xx, xx, zz;\n"
        "mov.b64 {%0, %1}, xx;\n"
        "}\n" : "=f"(y0), "=f"(y1) : "f"(x0), "f"(x1), "f"(z0), "f"(z1));
}
__device__ __forceinline__ void add2_f32(float x0, float x1, float& y0, float& y1) {
    asm("{\n"
        ".reg .b64 xx, yy;\n"
        "mov.b64 xx, {%2, %3};\n"
        "mov.b64 yy, {%0, %1};\n"
        "add.rn.f32x2 yy, yy, xx;\n"
        "mov.b64 {%0, %1}, yy;\n"
        "}\n" : "+f"(y0), "+f"(y1) : "f"(x0), "f"(x1));
}
// Four e4m3 bytes (lowest byte first) -> four floats.  Two hardware conversions to f16 pairs (exact: every e4m3 value is
// an f16 value), then to f32.
__device__ __forceinline__ void e4m3x4_to_f32(uint32_t w, float& f0, float& f1, float& f2, float& f3) {
    uint32_t h01, h23;
    asm("{\n"
        ".reg .b16 lo, hi;\n"
        "mov.b32 {lo, hi}, %2;\n"
        "cvt.rn.f16x2.e4m3x2 %0, lo;\n"
        "cvt.rn.f16x2.e4m3x2 %1, hi;\n"
        "}\n" : "=r"(h01), "=r"(h23) : "r"(w));
    asm("{\n"
        ".reg .b16 a, b;\n"
        "mov.b32 {a, b}, %2;\n"
        "cvt.f32.f16 %0, a;\n"
        "cvt.f32.f16 %1, b;\n"
        "}\n" : "=f"(f0), "=f"(f1) : "r"(h01));
    asm("{\n"
        ".reg .b16 a, b;\n"
        "mov.b32 {a, b}, %2;\n"
        "cvt.f32.f16 %0, a;\n"
        "cvt.f32.f16 %1, b;\n"
        "}\n" : "=f"(f2), "=f"(f3) : "r"(h23));
}
// x = hi + mid + lo with three bf16 values (3 x 8 significant bits: exact for every fp32 x whose parts stay normal);
// w01 = {hi, mid}, w2 = {lo, 0} as packed pairs, low half first.
__device__ __forceinline__ void split3_bf16(float x, uint32_t& w01, uint32_t& w2) {
    const uint32_t hi = pack_bf16x2(x, 0.f) & 0xffffu;
    const float r1 = x - __uint_as_float(hi << 16);
    const uint32_t mid = pack_bf16x2(r1, 0.f) & 0xffffu;
    const float r2 = r1 - __uint_as_float(mid << 16);
    const uint32_t lo = pack_bf16x2(r2, 0.f) & 0xffffu;
    w01 = hi | (mid << 16);
    w2 = lo;
}
__device__ __forceinline__ float bf16_lo_to_f32(uint32_t packed) { return __uint_as_float(packed << 16); }
__device__ __forceinline__ float bf16_hi_to_f32(uint32_t packed) { return __uint_as_float(packed & 0xffff0000u); }

}  // namespace moda

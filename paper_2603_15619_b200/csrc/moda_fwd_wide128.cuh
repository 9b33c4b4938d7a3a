// MoDA forward kernel, two softmax warpgroups at d = 128 (operator, boundary and data layout as in moda_fwd.cuh; the d = 64 form is in
// moda_fwd_wide.cuh).
//
// moda_fwd_kernel's pace is one warpgroup's softmax pass over a score tile: about 2000 cycles, with 1024 of the SFU for the
// exponentials and some 1500 for a warp that has its scheduler to itself beside the MMAs.  Two warpgroups on alternate key tiles overlap
// one's exponentials with the other's loads, maximum and stores -- but with P_j in the columns of S_j a score buffer is taken until PV_j
// completes, and O and the depth partial leave room for two: neither warpgroup finds its next tile ready (900 against 996 TFLOP/s).
// Here a warpgroup takes a whole score tile into registers at once (128 a thread) and P_j goes to columns of its own: the one score
// buffer can take S_{j+1} some 300 cycles after S_j was ready, and S_{j+1} is there when the other warpgroup asks for it.
// K tiles are loaded one ahead of V tiles: in the order K_j, V_j a K tile waits behind the V tile before it, whose stage is released by
// PV_{j-2}, and comes 1700 cycles late (T = 65536, 8 heads, l = 0: 8.15 ms so, 6.97 here, 8.77 moda_fwd_kernel).
//
// Cycles per key tile, T = 8192: 1620 (moda_fwd_kernel 2000); tensor cores 1024, exponentials 1150 with two warps on a scheduler.
// A warpgroup's pass was 2900 (load 180, maximum 440, agreeing on the reference and waiting for P_j's buffer 690, exponentials 1420, store 170),
// and S_j to S_{j+1} 1350 (load 180, hand-over 280, product 560, hand-over 280).  The reference read before the maximum and the buffer asked
// for behind it: 2-4 % faster; the reference read while the scores travel delays the hand-over by as much as it saves; the buffer asked
// for in front of the first store, or all stores behind the exponentials: 4-7 % slower.  us, in turn with moda_fwd_kernel: moda_api.cu,
// fwd_two_softmax.
//
// One CTA owns one (b, query head h) and one query tile or a pair of them (pair_coord), as in moda_fwd_kernel.  512 threads:
//
//   warps 0-3, 4-7   softmax A / B: one thread per query row in each; key tiles counted over the CTA's query tiles, A the even
//                    ones.  Both share one reference maximum per row (shared memory, published right after the maximum of each
//                    tile); O in tensor memory is rescaled only when it grows by more than 2^8.  Both run the epilogue, half
//                    of the features each.
//   warps 8-11       depth: as in moda_fwd_kernel, with e4m3 codes 64 features at a time as well (112 registers).
//   warp 12          TMA producer          warp 13   issues S_j = Q K_j^T; owns TMEM
//   warp 14          depth-cache producer  warp 15   issues O += P_j V_j
//
// TMEM columns (fp32): [0,128) S_j   [128,192), [192,256) P_j, even and odd j   [256,384) O   [384,512) o_d.
#pragma once

#include "moda_cache.cuh"
#include "moda_fwd.cuh"
#include "sm100_ptx.cuh"

namespace moda::d128 {

constexpr int kFwd2Threads = 512;   // four warpgroups: softmax A, softmax B, depth, {TMA, MMA S, depth producer, MMA PV}

// FP8: the depth cache holds e4m3 codes with a scale per row (moda_cache.cuh); the 128 row scales of a unit travel beside it.
template <bool FP8>
struct Fwd2Smem {
    static constexpr int D = 128;
    static constexpr int kTileBytes = kTileRows * D * 2;          // one 128 x D bf16 tile
    static constexpr int kSubBytes = kTileRows * 128;             // one 128 x 64 sub-tile
    static constexpr int kQ = 0;
    static constexpr int kK = kQ + kTileBytes;                    // 2 stages
    static constexpr int kV = kK + 2 * kTileBytes;                // 2 stages
    static constexpr int kU = kV + 2 * kTileBytes;                // depth scores [32][128] fp32
    static constexpr int kMd = kU + 32 * kTileRows * 4;           // m_d [128], l_d [128]
    static constexpr int kMref = kMd + 2 * kTileRows * 4;         // reference maximum [128], shared by the two softmax warpgroups
    static constexpr int kLx = kMref + kTileRows * 4;             // row sums [128], exchanged in the epilogue
    static constexpr int kRing = kLx + kTileRows * 4;             // depth units: 64 features of one slot's keys (values)
    static constexpr int kUnitBytes = FP8 ? 64 * kTileRows : 8 * kTileRows * 16;  // 16 KiB (e4m3: 8 KiB), contiguous in the cache
    static constexpr int kScaleBytes = FP8 ? kTileRows * 4 : 0;   // row scales of a unit
    static constexpr int kNumBars = 34;
    static constexpr int kSmemLimit = 232448;                     // 227 KiB per CTA on sm_100
    // no slack for aligning the segment by hand (the ring needs it): it is declared 1024-aligned and checked at run time
    static constexpr int kRingFit = (kSmemLimit - kRing - kNumBars * 8 - 16) / (kUnitBytes + kScaleBytes);
    static constexpr int kRingStages = kRingFit < 6 ? kRingFit : 6;   // every unit that fits, at most 6
    static_assert(kRingStages >= 3, "depth ring too shallow");
    static constexpr int kScale = kRing + kRingStages * kUnitBytes;   // [ring stage][128] fp32 (e4m3 only)
    static constexpr int kBars = kScale + kRingStages * kScaleBytes;
    static constexpr int kMisc = kBars + kNumBars * 8;            // tmem base, abort flag
    static constexpr int kTotal = kMisc + 16;
    static constexpr int kDynamic = kTotal;
};

enum Fwd2Bar : int {
    kBarQ = 0,
    kBarKFull = 1,    // +stage
    kBarVFull = 5,    // +stage
    kBarVEmpty = 7,   // +stage: PV_j complete (V stage and P buffer free; O may be rescaled)
    kBarSFull = 9,    // +(jj & 1): S_j complete (also frees the K stage)
    kBarPFull = 11,   // +P buffer
    kBarDrain2 = 13,  // abort path of the second issuer
    kBarDepth = 14,
    kBarOFinal = 15,  // one phase per query tile: every MMA of the tile has completed
    kBarDrain = 16,
    kBarDFull = 17,   // +ring stage (<= 6): depth unit landed
    kBarDEmpty = 23,  // +ring stage (<= 6): all 128 depth threads have read the unit
    kBarRef = 29,     // +(jj & 1): the reference maximum for key tile jj has been published
    kBarXFree = 31,   // S_j is in registers: the score buffer may take S_{j+1}
    kBarTileDone = 32,  // one phase per query tile of the CTA: its epilogue (output stored) is complete
};

template <bool FP8>
__global__ void __launch_bounds__(kFwd2Threads, 1)
moda_fwd2_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapO,
                const FwdParams p) {
    using L = Fwd2Smem<FP8>;
    constexpr int D = L::D;
    constexpr int NSUB = D / 64;
    constexpr uint32_t kTmemCols = 512;
    constexpr uint32_t kColP = 128, kColO = 256, kColOd = 384;

    if (g_moda_status != 0) return;   // an earlier kernel gave up a wait: do not pile up more timeouts

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = aligned_dynamic_smem(smem_raw, L::kTotal);
    if (smem == nullptr) {
        if (threadIdx.x == 0) atomicCAS(&g_moda_status, 0, kStatusSmemLayout);
        return;
    }
    const uint32_t sbase = smem_u32(smem);
    float* sU = reinterpret_cast<float*>(smem + L::kU);
    float* sMd = reinterpret_cast<float*>(smem + L::kMd);
    float* sLd = sMd + kTileRows;
    float* sMref = reinterpret_cast<float*>(smem + L::kMref);
    float* sLx = reinterpret_cast<float*>(smem + L::kLx);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kMisc + 4);
    auto bar = [&](int i) { return sbase + L::kBars + 8u * uint32_t(i); };

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;

    const int nq = num_tiles(p.T);
    const bool paired = p.pair != 0;
    const TileCoord tc = paired ? pair_coord(blockIdx.x, nq, p.H, p.G) : tile_coord(blockIdx.x, nq, p.H, p.G);
    const int b = tc.b, h = tc.h, hk = tc.hk;
    const int Hk = p.H / p.G;
    // the CTA's query tiles, the longer one first; every role walks them in this order
    const int n_tiles = (paired && nq - 1 - tc.qt != tc.qt) ? 2 : 1;
    auto tile_qt = [&](int t) { return (paired && t == 0) ? nq - 1 - tc.qt : tc.qt; };
    // causal: key tiles up to the one that holds the last row's own position (row i sees keys <= i + kv_off)
    auto tile_nkv = [&](int t) {
        return min((tile_qt(t) * kTileRows + kTileRows + p.kv_off + kTileRows - 1) / kTileRows, num_tiles(p.T_kv));
    };

    if (tid == 0) {
        *abort_flag = 0;
        mbar_init(bar(kBarQ), 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar(kBarKFull + s), 1);
            mbar_init(bar(kBarVFull + s), 1);
            mbar_init(bar(kBarVEmpty + s), 1);
            mbar_init(bar(kBarSFull + s), 1);
            mbar_init(bar(kBarPFull + s), 128);
        }
        for (int s = 0; s < 2; ++s) mbar_init(bar(kBarRef + s), 128);
        mbar_init(bar(kBarXFree), 128);
        mbar_init(bar(kBarDepth), 128);
        mbar_init(bar(kBarTileDone), 1);
        mbar_init(bar(kBarOFinal), 1);
        mbar_init(bar(kBarDrain), 1);
        mbar_init(bar(kBarDrain2), 1);
        for (int s = 0; s < L::kRingStages; ++s) {
            mbar_init(bar(kBarDFull + s), 1);
            mbar_init(bar(kBarDEmpty + s), 128);
        }
        fence_mbar_init();
    }
    if (warp == 13) {
        tmem_alloc(smem_u32(tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    // Register budget: the launch gives every warp 128 registers; the depth and the producer warpgroup hand on what they do not need.
    // 176 / 112 / 48 against 168 / 120 / 56: 1 % faster; with 104 or 96 for the depth warps they spill (short sequences 5 % slower).
    constexpr int kRegsSoftmax = 176, kRegsDepth = 112, kRegsProducer = 48;
    static_assert(2 * kRegsSoftmax + kRegsDepth + kRegsProducer <= 4 * 128, "register shares of the four warpgroups");
    if (warp < 8) {
        // =========================== softmax A / B + epilogue ===========================
        setmaxnreg_inc<kRegsSoftmax>();
        const int wg = warp >> 2;                        // 0: even key tiles (counted over the CTA's query tiles), 1: odd ones
        const int r = tid & 127;                         // query row inside the tile = TMEM lane
        const uint32_t lane_addr = uint32_t((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + lane_addr, tP = tS + kColP + wg * 64;
        int jbase = 0;                                   // key tiles of the CTA's earlier query tiles: the rings run on
#pragma unroll 1
        for (int t = 0; t < n_tiles; ++t) {
        const int qt = tile_qt(t), q0 = qt * kTileRows, n_kv = tile_nkv(t);
        float my_ref = -INFINITY;                        // reference maximum (log2 domain) that l_part is expressed in
        float l_part = 0.f;                              // this warpgroup's share of the row sum
#pragma unroll 1
        for (int j = (jbase ^ wg) & 1; j < n_kv; j += 2) {
            const int jj = jbase + j;                    // jj & 1 == wg: barriers and P buffer of that parity are this warpgroup's
            mbar_wait(bar(kBarSFull + wg), (jj >> 1) & 1, abort_flag, 10);
            tc_fence_after_sync();
            uint32_t sv[4][32];
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld32(tS + c * 32, sv[c]);
            tmem_wait_ld();
            tc_fence_before_sync();
            mbar_arrive(bar(kBarXFree));                 // the score buffer may take S_{j+1}
            // the reference maximum that the other warpgroup has chosen for the key tile before: its way here passes under the maximum below
            float m_prev = -INFINITY;
            if (j > 0) {
                mbar_wait(bar(kBarRef + (wg ^ 1)), ((jj - 1) >> 1) & 1, abort_flag, 14);
                m_prev = sMref[r];
            }
            if ((j + 1) * kTileRows - 1 > q0 + p.kv_off) {   // tile reaches past the first row's position: causal mask
                const int rs = r + q0 + p.kv_off - j * kTileRows;   // column i of this tile is visible iff i <= rs
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (c * 32 + i > rs) sv[c][i] = 0xff800000u;
            }
            float mx[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
                for (int i = 0; i < 32; i += 4) {        // 3-input max: one instruction per two scores
                    m0 = max3(m0, __uint_as_float(sv[c][i]), __uint_as_float(sv[c][i + 1]));
                    m1 = max3(m1, __uint_as_float(sv[c][i + 2]), __uint_as_float(sv[c][i + 3]));
                }
                mx[c] = fmaxf(m0, m1);
            }
            const float tile_max = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * p.scale_log2;
            // ---- agree on the reference maximum with the other warpgroup ----
            const float m_new = fmaxf(m_prev, tile_max);
            // j == 0: nothing accumulated yet, adopt the tile maximum.  Later: move the reference only
            // when some row of this warp grew by more than the threshold (decision per warp, because
            // the TMEM accesses of the rescale are warp-wide).
            const bool move = (j == 0) || __any_sync(0xffffffffu, m_new - m_prev > kRescaleThreshold);
            const float m_ref = move ? m_new : m_prev;
            sMref[r] = m_ref;
            mbar_arrive(bar(kBarRef + wg));              // tile j+1 may now pick its reference
            if (jj >= 2) mbar_wait(bar(kBarVEmpty + wg), ((jj - 2) >> 1) & 1, abort_flag, 17);   // PV_{j-2} has read the buffer that P_j goes to
            if (move && j > 0) {
                // The maximum grew a lot: bring O to the new reference.  O may only be touched between PV_{j-1}
                // completing and PV_j being issued; PV_j waits for this thread's arrival on kBarPFull below.  (The barrier's
                // phase before that one, PV_{j-3}, has completed: PV_{j-2} has, see above.)
                mbar_wait(bar(kBarVEmpty + (wg ^ 1)), ((jj - 1) >> 1) & 1, abort_flag, 11);
                tc_fence_after_sync();
                const float f = fast_exp2(m_prev - m_ref);
#pragma unroll 1                                             // rare: kept small (unrolled, this branch cost every tile 2 %)
                for (int c = 0; c < D / 16; ++c) {
                    uint32_t o[16];
                    tmem_ld16(tmem + lane_addr + kColO + c * 16, o);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
                    tmem_st16(tmem + lane_addr + kColO + c * 16, o);
                }
            }
            if (my_ref != m_ref) {                       // re-express this warpgroup's partial sum
                l_part *= fast_exp2(my_ref - m_ref);     // (first tile: 0 * exp2(-inf) = 0)
                my_ref = m_ref;
            }
            const float neg_m = -m_ref;
            tc_fence_after_sync();
            // Packed fp32 FMAs and additions: the pipes take as long for them as for twice as many scalar ones, but a tile takes
            // 128 instructions fewer.  Four sums here, four in the other warpgroup.
            float sum0 = 0.f, sum1 = 0.f, sum2 = 0.f, sum3 = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t pk[16];
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                    float a0, a1, b0, b1;
                    fma2_scale(__uint_as_float(sv[c][2 * i]), __uint_as_float(sv[c][2 * i + 1]), p.scale_log2, neg_m, a0, a1);
                    fma2_scale(__uint_as_float(sv[c][2 * i + 2]), __uint_as_float(sv[c][2 * i + 3]), p.scale_log2, neg_m, b0, b1);
                    a0 = fast_exp2(a0);
                    a1 = fast_exp2(a1);
                    b0 = fast_exp2(b0);
                    b1 = fast_exp2(b1);
                    add2_f32(a0, a1, sum0, sum1);
                    add2_f32(b0, b1, sum2, sum3);
                    pk[i] = pack_bf16x2(a0, a1);
                    pk[i + 1] = pack_bf16x2(b0, b1);
                }
                tmem_st16(tP + c * 16, pk);
            }
            l_part += (sum0 + sum1) + (sum2 + sum3);
            tmem_wait_st();
            tc_fence_before_sync();
            mbar_arrive(bar(kBarPFull + wg));
        }

        // ------------------------------ epilogue ------------------------------
        // Final reference = the one published for the last key tile; the warpgroups add their partial sums (in that
        // reference) through shared memory.
        const int last = jbase + n_kv - 1;
        mbar_wait(bar(kBarRef + (last & 1)), (last >> 1) & 1, abort_flag, 15);
        const float m_ref = sMref[r];
        if (my_ref != m_ref) l_part = (my_ref == -INFINITY) ? 0.f : l_part * fast_exp2(my_ref - m_ref);
        if (wg == 1) sLx[r] = l_part;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        float l_sum = l_part;
        if (wg == 0) {                                   // row r of A is the only other user of sLx[r]
            l_sum += sLx[r];
            sLx[r] = l_sum;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (wg == 1) l_sum = sLx[r];

        mbar_wait(bar(kBarOFinal), t & 1, abort_flag, 12);
        tc_fence_after_sync();
        float a_s = 1.f, a_d = 0.f, m_fin = m_ref, l_fin = l_sum;
        if (p.l > 0) {
            mbar_wait(bar(kBarDepth), t & 1, abort_flag, 13);
            tc_fence_after_sync();
            const float m_d = sMd[r], l_d = sLd[r];
            m_fin = fmaxf(m_ref, m_d);
            a_s = fast_exp2(m_ref - m_fin);
            a_d = fast_exp2(m_d - m_fin);
            l_fin = a_s * l_sum + a_d * l_d;
        }
        const float inv = 1.f / l_fin;
        a_s *= inv;
        a_d *= inv;
        // O tile -> shared memory (the Q buffer, in the same swizzled layout) -> TMA store.
#pragma unroll
        for (int cc = 0; cc < D / 64; ++cc) {            // half of the feature columns each
            const int c = wg * (D / 64) + cc;
            uint32_t o[32];
            tmem_ld32(tmem + lane_addr + kColO + c * 32, o);
            tmem_wait_ld();
            float of[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) of[i] = __uint_as_float(o[i]) * a_s;
            if (p.l > 0) {
                uint32_t od[32];
                tmem_ld32(tmem + lane_addr + kColOd + c * 32, od);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) of[i] = fmaf(__uint_as_float(od[i]), a_d, of[i]);
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                uint4 v;
                v.x = pack_bf16x2(of[8 * g + 0], of[8 * g + 1]);
                v.y = pack_bf16x2(of[8 * g + 2], of[8 * g + 3]);
                v.z = pack_bf16x2(of[8 * g + 4], of[8 * g + 5]);
                v.w = pack_bf16x2(of[8 * g + 6], of[8 * g + 7]);
                *reinterpret_cast<uint4*>(smem + L::kQ + swz_chunk_offset(r, c * 4 + g)) = v;
            }
        }
        if (wg == 0 && q0 + r < p.T) p.LSE[(size_t(b) * p.H + h) * p.T + q0 + r] = (m_fin + log2f(l_fin)) * kLn2;
        fence_proxy_async_smem();
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (tid == 0) {
#pragma unroll
            for (int s = 0; s < NSUB; ++s)
                tma_store_4d(&mapO, sbase + L::kQ + s * L::kSubBytes, s * 64, h, q0, b);
            tma_store_commit();
            tma_store_wait_read();
        }
        // The tile is done: the Q buffer (output staging), O and the depth partial in tensor memory may be reused for the
        // CTA's next tile.
        tc_fence_before_sync();
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (tid == 0) mbar_arrive(bar(kBarTileDone));
        jbase += n_kv;
        }
    } else if (warp < 12) {
        // =========================== depth partial state ===========================
        setmaxnreg_dec<kRegsDepth>();
        if (p.l > 0) {
            const int r = tid - 256;
            const uint32_t lane_addr = uint32_t((warp & 3) * 32) << 16;
            int unit = 0;                                 // running index into the producer's unit sequence (over all tiles)
            // Reads this thread's 8 x 16 bytes of the next depth unit from the ring and frees the stage.
            auto take_unit = [&](uint4 (&dst)[8]) {
                const int st = unit % L::kRingStages;
                mbar_wait(bar(kBarDFull + st), (unit / L::kRingStages) & 1, abort_flag, 21);
                const uint8_t* src = smem + L::kRing + st * L::kUnitBytes + r * 16;
#pragma unroll
                for (int c = 0; c < 8; ++c) dst[c] = *reinterpret_cast<const uint4*>(src + c * (kTileRows * 16));
                // The stage is refilled by the async proxy (bulk copy) while these loads went through the
                // generic proxy: the proxy fence orders them before the refill that this arrival allows.
                fence_proxy_async_smem();
                mbar_arrive(bar(kBarDEmpty + st));
                ++unit;
            };
            // The slots are handled in groups of kFwdDepthGroup (the score scratch holds one group): an
            // online softmax over the groups, with the partial output o_d rescaled in TMEM when a later
            // group raises the maximum.  Up to 32 slots are one group.
#pragma unroll 1
            for (int t = 0; t < n_tiles; ++t) {
            const int qt = tile_qt(t), q0 = qt * kTileRows;
            // this thread's query row (zeros past T, as the TMA-loaded tile has them)
            const bool qvalid = q0 + r < p.T;
            const uint4* qrow = reinterpret_cast<const uint4*>(p.Q + ((size_t(b) * p.T + (qvalid ? q0 + r : 0)) * p.H + h) * D);
            // The depth partial of the CTA's previous tile stays parked (tensor memory, sMd / sLd) until that tile's
            // epilogue has read it; this tile's slots are streamed and used meanwhile, only the first store waits.
            auto wait_previous_tile = [&]() { if (t > 0) mbar_wait(bar(kBarTileDone), (t - 1) & 1, abort_flag, 25); };
            float m_d = -INFINITY, l_d = 0.f;
            if constexpr (FP8) {
                // e4m3 cache: a unit holds 64 features of one slot's keys (values) for the tile's rows, its row
                // scales sit beside it; codes are widened to fp32 in registers, everything else as below.  Packed fp32 FMAs
                // (T = 8192, B = 2, 16 heads, us: l = 8 694 -> 670, l = 16 793 -> 732, l = 32 972 -> 859).
                const float* sScale = reinterpret_cast<const float*>(smem + L::kScale);
                auto take_unit8 = [&](uint4 (&dst)[4], float& sc) {
                    const int st = unit % L::kRingStages;
                    mbar_wait(bar(kBarDFull + st), (unit / L::kRingStages) & 1, abort_flag, 21);
                    const uint8_t* src = smem + L::kRing + st * L::kUnitBytes + r * 16;
#pragma unroll
                    for (int c = 0; c < 4; ++c) dst[c] = *reinterpret_cast<const uint4*>(src + c * (kTileRows * 16));
                    sc = sScale[st * kTileRows + r];
                    fence_proxy_async_smem();
                    mbar_arrive(bar(kBarDEmpty + st));
                    ++unit;
                };
#pragma unroll 1
                for (int g0 = 0; g0 < p.l; g0 += kFwdDepthGroup) {
                    const int gl = min(kFwdDepthGroup, p.l - g0);
                    // ---- depth scores u_i = s_i <q, codes_i>, 64 features per sweep ----
#pragma unroll 1
                    for (int half = 0; half < NSUB; ++half) {
                        float q[64];
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            const uint4 v = qvalid ? __ldg(qrow + half * 8 + c) : make_uint4(0u, 0u, 0u, 0u);
                            q[8 * c + 0] = bf16_lo_to_f32(v.x); q[8 * c + 1] = bf16_hi_to_f32(v.x);
                            q[8 * c + 2] = bf16_lo_to_f32(v.y); q[8 * c + 3] = bf16_hi_to_f32(v.y);
                            q[8 * c + 4] = bf16_lo_to_f32(v.z); q[8 * c + 5] = bf16_hi_to_f32(v.z);
                            q[8 * c + 6] = bf16_lo_to_f32(v.w); q[8 * c + 7] = bf16_hi_to_f32(v.w);
                        }
#pragma unroll 1
                        for (int i = 0; i < gl; ++i) {
                            uint4 cur[4];
                            float sc;
                            take_unit8(cur, sc);
                            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const uint32_t w[4] = {cur[c].x, cur[c].y, cur[c].z, cur[c].w};
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    float f0, f1, f2, f3;
                                    e4m3x4_to_f32(w[k], f0, f1, f2, f3);
                                    fma2_f32(q[16 * c + 4 * k + 0], q[16 * c + 4 * k + 1], f0, f1, a0, a1);
                                    fma2_f32(q[16 * c + 4 * k + 2], q[16 * c + 4 * k + 3], f2, f3, a2, a3);
                                }
                            }
                            const float part = ((a0 + a1) + (a2 + a3)) * sc;
                            if (half == 0) sU[i * kTileRows + r] = part;
                            else sU[i * kTileRows + r] += part;
                        }
                    }
                    float m_new = m_d;
#pragma unroll 1
                    for (int i = 0; i < gl; ++i) m_new = fmaxf(m_new, sU[i * kTileRows + r] * p.scale_log2);
                    const float f = fast_exp2(m_d - m_new);       // first group: exp2(-inf) = 0
                    l_d *= f;
#pragma unroll 1
                    for (int i = 0; i < gl; ++i) {
                        const float w = fast_exp2(fmaf(sU[i * kTileRows + r], p.scale_log2, -m_new));
                        sU[i * kTileRows + r] = w;
                        l_d += w;
                    }
                    m_d = m_new;
                    // ---- o_d = sum_i (w_i s_i) codes_i, 64 features per sweep, parked in TMEM ----
#pragma unroll 1
                    for (int half = 0; half < NSUB; ++half) {
                        float acc[64];
                        if (g0 == 0) {
#pragma unroll
                            for (int c = 0; c < 64; ++c) acc[c] = 0.f;
                        } else {
#pragma unroll
                            for (int c = 0; c < 2; ++c) {
                                uint32_t o[32];
                                tmem_ld32(tmem + lane_addr + kColOd + half * 64 + c * 32, o);
                                tmem_wait_ld();
#pragma unroll
                                for (int i = 0; i < 32; ++i) acc[32 * c + i] = __uint_as_float(o[i]) * f;
                            }
                        }
#pragma unroll 1
                        for (int i = 0; i < gl; ++i) {
                            uint4 cur[4];
                            float sc;
                            take_unit8(cur, sc);
                            const float w = sU[i * kTileRows + r] * sc;
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const uint32_t ww[4] = {cur[c].x, cur[c].y, cur[c].z, cur[c].w};
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    float f0, f1, f2, f3;
                                    e4m3x4_to_f32(ww[k], f0, f1, f2, f3);
                                    fma2_f32(w, w, f0, f1, acc[16 * c + 4 * k + 0], acc[16 * c + 4 * k + 1]);
                                    fma2_f32(w, w, f2, f3, acc[16 * c + 4 * k + 2], acc[16 * c + 4 * k + 3]);
                                }
                            }
                        }
                        if (g0 == 0 && half == 0) wait_previous_tile();
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            uint32_t o[32];
#pragma unroll
                            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(acc[32 * c + i]);
                            tmem_st32(tmem + lane_addr + kColOd + half * 64 + c * 32, o);
                        }
                        tmem_wait_st();                          // a later group reads these columns back
                    }
                }
            } else {
#pragma unroll 1
            for (int g0 = 0; g0 < p.l; g0 += kFwdDepthGroup) {
                const int gl = min(kFwdDepthGroup, p.l - g0);
                // ---- depth scores u_i = <q, kd_i>, 64 features per sweep ----
#pragma unroll 1
                for (int half = 0; half < NSUB; ++half) {
                    uint4 q[8];                              // stays packed: the products are mixed-precision FMAs
#pragma unroll
                    for (int c = 0; c < 8; ++c) q[c] = qvalid ? __ldg(qrow + half * 8 + c) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
                    for (int i = 0; i < gl; ++i) {
                        uint4 cur[8];
                        take_unit(cur);
                        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            fma2_bf16x2(q[c].x, cur[c].x, a0, a1);
                            fma2_bf16x2(q[c].y, cur[c].y, a2, a3);
                            fma2_bf16x2(q[c].z, cur[c].z, a0, a1);
                            fma2_bf16x2(q[c].w, cur[c].w, a2, a3);
                        }
                        const float part = (a0 + a1) + (a2 + a3);
                        if (half == 0) sU[i * kTileRows + r] = part;
                        else sU[i * kTileRows + r] += part;
                    }
                }
                // ---- partial softmax over the depth scores seen so far ----
                float m_new = m_d;
#pragma unroll 1
                for (int i = 0; i < gl; ++i) m_new = fmaxf(m_new, sU[i * kTileRows + r] * p.scale_log2);
                const float f = fast_exp2(m_d - m_new);       // first group: exp2(-inf) = 0
                l_d *= f;
#pragma unroll 1
                for (int i = 0; i < gl; ++i) {
                    const float w = fast_exp2(fmaf(sU[i * kTileRows + r], p.scale_log2, -m_new));
                    sU[i * kTileRows + r] = w;
                    l_d += w;
                }
                m_d = m_new;
                // ---- o_d = sum_i w_i vd_i, 64 features per sweep, parked in TMEM ----
#pragma unroll 1
                for (int half = 0; half < NSUB; ++half) {
                    float acc[64];
                    if (g0 == 0) {
#pragma unroll
                        for (int c = 0; c < 64; ++c) acc[c] = 0.f;
                    } else {
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            uint32_t o[32];
                            tmem_ld32(tmem + lane_addr + kColOd + half * 64 + c * 32, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < 32; ++i) acc[32 * c + i] = __uint_as_float(o[i]) * f;
                        }
                    }
#pragma unroll 1
                    for (int i = 0; i < gl; ++i) {
                        uint4 cur[8];
                        take_unit(cur);
                        const float w = sU[i * kTileRows + r];
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            axpy_bf16x2(w, cur[c].x, acc[8 * c + 0], acc[8 * c + 1]);
                            axpy_bf16x2(w, cur[c].y, acc[8 * c + 2], acc[8 * c + 3]);
                            axpy_bf16x2(w, cur[c].z, acc[8 * c + 4], acc[8 * c + 5]);
                            axpy_bf16x2(w, cur[c].w, acc[8 * c + 6], acc[8 * c + 7]);
                        }
                    }
                    if (g0 == 0 && half == 0) wait_previous_tile();
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t o[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(acc[32 * c + i]);
                        tmem_st32(tmem + lane_addr + kColOd + half * 64 + c * 32, o);
                    }
                    tmem_wait_st();                          // a later group reads these columns back
                }
            }
            }
            sMd[r] = m_d;
            sLd[r] = l_d;
            tmem_wait_st();
            tc_fence_before_sync();
            mbar_arrive(bar(kBarDepth));
            }
        }
        if (!FP8 && p.append_slot != nullptr && h == hk * p.G) {
            // the write step: every read of the depth cache by this CTA is complete here, so the slot may be one that was read
#pragma unroll 1
            for (int t = 0; t < n_tiles; ++t)
                append_rows_from_global<D>(p.append_slot, p.K, p.V, b, hk, Hk, p.T, nq, tile_qt(t), tid - 256);
        }
    } else {
      setmaxnreg_dec<kRegsProducer>();   // one instruction for the whole producer warpgroup (warps 12-15)
      if (warp == 12) {
        // =========================== TMA producer ===========================
        if (lane == 0) {
            tma_prefetch_desc(&mapQ);
            tma_prefetch_desc(&mapK);
            tma_prefetch_desc(&mapV);
            // K tiles run one ahead of V tiles: K_{j+1} only waits for S_{j-1} (its stage's last tile), V_j for PV_{j-2}, which comes later.
            auto load_K = [&](int jj, int j) {
                const int kst = jj & 1;
                if (jj >= 2) mbar_wait(bar(kBarSFull + kst), ((jj - 2) >> 1) & 1, abort_flag, 30);   // S of the stage's last tile is complete
                mbar_arrive_expect_tx(bar(kBarKFull + kst), L::kTileBytes);
#pragma unroll
                for (int s = 0; s < NSUB; ++s)
                    tma_load_4d(sbase + L::kK + kst * L::kTileBytes + s * L::kSubBytes, &mapK, bar(kBarKFull + kst), s * 64, hk, j * kTileRows, b);
            };
            int jbase = 0;
#pragma unroll 1
            for (int t = 0; t < n_tiles; ++t) {
                const int q0 = tile_qt(t) * kTileRows, n_kv = tile_nkv(t);
                if (t > 0) mbar_wait(bar(kBarTileDone), (t - 1) & 1, abort_flag, 33);
                mbar_arrive_expect_tx(bar(kBarQ), L::kTileBytes);
#pragma unroll
                for (int s = 0; s < NSUB; ++s)
                    tma_load_4d(sbase + L::kQ + s * L::kSubBytes, &mapQ, bar(kBarQ), s * 64, h, q0, b);
                if (t == 0) load_K(0, 0);
#pragma unroll 1
                for (int j = 0; j < n_kv; ++j) {
                    const int jj = jbase + j, st = jj & 1;
                    if (j + 1 < n_kv) load_K(jj + 1, j + 1);
                    else if (t + 1 < n_tiles) load_K(jj + 1, 0);
                    if (jj >= 2) mbar_wait(bar(kBarVEmpty + st), ((jj - 2) >> 1) & 1, abort_flag, 31);
                    mbar_arrive_expect_tx(bar(kBarVFull + st), L::kTileBytes);
#pragma unroll
                    for (int s = 0; s < NSUB; ++s)
                        tma_load_4d(sbase + L::kV + st * L::kTileBytes + s * L::kSubBytes, &mapV, bar(kBarVFull + st),
                                    s * 64, hk, j * kTileRows, b);
                }
                jbase += n_kv;
            }
        }
      } else if (warp == 13) {
        // =========================== MMA issuer: S_j = Q K_j^T ===========================
        {   // whole warp: operands are warp-uniform, one elected lane issues
            constexpr uint32_t idesc_s = make_idesc_bf16(128, 128, false, false);
            // every descriptor is built once; inside the loop a descriptor is one 64-bit add (the
            // start-address field counts 16-byte units and stays inside its 14 bits below 256 KiB)
            uint64_t dq[D / 16];
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) dq[kk] = desc_kmajor_sw128(sbase + L::kQ + (kk >> 2) * L::kSubBytes, kk & 3);
            const uint64_t dk0 = desc_kmajor_sw128(sbase + L::kK, 0);
            int jbase = 0;
#pragma unroll 1
            for (int t = 0; t < n_tiles; ++t) {
            const int n_kv = tile_nkv(t);
            mbar_wait(bar(kBarQ), t & 1, abort_flag, 41);
#pragma unroll 1
            for (int j = 0; j < n_kv; ++j) {
                const int jj = jbase + j;
                const int kst = jj & 1;
                // the score buffer still holds S_{j-1} until it is in registers
                if (jj >= 1) mbar_wait2(bar(kBarKFull + kst), (jj >> 1) & 1, bar(kBarXFree), (jj - 1) & 1, abort_flag, 40, 44);
                else mbar_wait(bar(kBarKFull + kst), 0, abort_flag, 40);
                tc_fence_after_sync();
                const uint64_t dk = dk0 + uint64_t((kst * L::kTileBytes) >> 4);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk)
                    umma_ss(tmem, dq[kk], dk + uint64_t(((kk >> 2) * L::kSubBytes + (kk & 3) * 32) >> 4), idesc_s, kk > 0);
                umma_commit(bar(kBarSFull + (jj & 1)));
            }
            jbase += n_kv;
            }
            if (*abort_flag != 0) {
                // A wait gave up somewhere: make sure no MMA of this thread is still in flight before TMEM is released.
                umma_commit(bar(kBarDrain));
                const uint64_t t0 = globaltimer_ns();
                while (!mbar_try_wait(bar(kBarDrain), 0) && globaltimer_ns() - t0 < 20000000ull) {}
            }
        }
      } else if (warp == 15) {
        // =========================== MMA issuer: O += P_j V_j ===========================
        {   // whole warp: operands are warp-uniform, one elected lane issues
            constexpr uint32_t idesc_o = make_idesc_bf16(128, D, false, true);
            const uint64_t dv0 = desc_mnmajor_sw128(sbase + L::kV, 0, L::kSubBytes);
            int jbase = 0;
#pragma unroll 1
            for (int t = 0; t < n_tiles; ++t) {
            const int n_kv = tile_nkv(t);
#pragma unroll 1
            for (int j = 0; j < n_kv; ++j) {
                const int jj = jbase + j;
                const int st = jj & 1;
                mbar_wait2(bar(kBarVFull + st), (jj >> 1) & 1, bar(kBarPFull + st), (jj >> 1) & 1, abort_flag, 42, 43);
                tc_fence_after_sync();
                const uint64_t dv = dv0 + uint64_t((st * L::kTileBytes) >> 4);
                const uint32_t tp = tmem + kColP + uint32_t(st) * 64u;
                umma_ts(tmem + kColO, tp, dv, idesc_o, j > 0);
#pragma unroll
                for (int kk = 1; kk < kTileRows / 16; ++kk)
                    umma_ts(tmem + kColO, tp + kk * 8, dv + uint64_t(kk * 128), idesc_o, 1);
                umma_commit(bar(kBarVEmpty + st));
            }
            // All S MMAs of the tile completed before the P they fed was written, so its last PV is its last MMA.
            umma_commit(bar(kBarOFinal));
            jbase += n_kv;
            }
            if (*abort_flag != 0) {
                // A wait gave up somewhere: make sure no MMA is still in flight before TMEM is released.
                umma_commit(bar(kBarDrain2));
                const uint64_t t0 = globaltimer_ns();
                while (!mbar_try_wait(bar(kBarDrain2), 0) && globaltimer_ns() - t0 < 20000000ull) {}
            }
        }
      } else if (warp == 14) {
        // =========================== depth-cache producer ===========================
        // Streams the tile's depth keys, then values, as 16 KiB units (8 feature chunks of one slot:
        // one contiguous run of the cache) through the ring, in the order the depth warps consume
        // them.  The ring keeps up to kRingStages x 16 KiB of HBM reads in flight per SM.
        if (FP8 && lane == 0 && p.l > 0) {
            // e4m3 cache: one unit per (slot, K or V): the block's codes, and its 128 row scales behind them
            const uint64_t policy = l2_policy_evict_first();
            const size_t slot_bytes = cache8_slot_bytes(p.B, p.T, Hk, D);
            const size_t blk_bytes = cache8_block_bytes(D);
            int unit = 0;
#pragma unroll 1
            for (int t = 0; t < n_tiles; ++t) {
            const uint8_t* blk = reinterpret_cast<const uint8_t*>(p.depth_kv) + (((size_t(b) * Hk + hk) * nq + tile_qt(t)) * 2) * blk_bytes;
#pragma unroll 1
            for (int g0 = 0; g0 < p.l; g0 += kFwdDepthGroup) {
                const int gl = min(kFwdDepthGroup, p.l - g0);
#pragma unroll 1
                for (int kv = 0; kv < 2; ++kv)
#pragma unroll 1
                    for (int half = 0; half < NSUB; ++half)
#pragma unroll 1
                        for (int i = 0; i < gl; ++i, ++unit) {
                            const int st = unit % L::kRingStages;
                            if (unit >= L::kRingStages)
                                mbar_wait(bar(kBarDEmpty + st), ((unit / L::kRingStages) - 1) & 1, abort_flag, 32);
                            mbar_arrive_expect_tx(bar(kBarDFull + st), L::kUnitBytes + L::kScaleBytes);
                            const uint8_t* src = blk + size_t(g0 + i) * slot_bytes + size_t(kv) * blk_bytes;
                            bulk_load(sbase + L::kRing + st * L::kUnitBytes, src + half * L::kUnitBytes, L::kUnitBytes, bar(kBarDFull + st), policy);
                            bulk_load(sbase + L::kScale + st * L::kScaleBytes, src + NSUB * L::kUnitBytes, L::kScaleBytes, bar(kBarDFull + st), policy);
                        }
            }
            }
        } else if (lane == 0 && p.l > 0) {
            const uint64_t policy = l2_policy_evict_first();          // the depth cache is read exactly once
            const size_t slot_bytes = cache_slot_elems(p.B, p.T, Hk, D) * 2;
            int unit = 0;
#pragma unroll 1
            for (int t = 0; t < n_tiles; ++t) {
            const uint8_t* blk = reinterpret_cast<const uint8_t*>(p.depth_kv) +
                                 (((size_t(b) * Hk + hk) * nq + tile_qt(t)) * 2) * (size_t(kTileRows) * D * 2);
#pragma unroll 1
            for (int g0 = 0; g0 < p.l; g0 += kFwdDepthGroup) {
                const int gl = min(kFwdDepthGroup, p.l - g0);
#pragma unroll 1
                for (int kv = 0; kv < 2; ++kv)
#pragma unroll 1
                    for (int half = 0; half < NSUB; ++half)
#pragma unroll 1
                        for (int i = 0; i < gl; ++i, ++unit) {
                            const int st = unit % L::kRingStages;
                            if (unit >= L::kRingStages)
                                mbar_wait(bar(kBarDEmpty + st), ((unit / L::kRingStages) - 1) & 1, abort_flag, 32);
                            mbar_arrive_expect_tx(bar(kBarDFull + st), L::kUnitBytes);
                            bulk_load(sbase + L::kRing + st * L::kUnitBytes,
                                      blk + size_t(g0 + i) * slot_bytes + size_t(kv) * (size_t(kTileRows) * D * 2) + size_t(half) * L::kUnitBytes,
                                      L::kUnitBytes, bar(kBarDFull + st), policy);
                        }
            }
            }
        }
      }
    }

    tc_fence_before_sync();
    __syncthreads();
    abort_teardown(abort_flag, 384);
    __syncthreads();
    if (warp == 13) tmem_dealloc(tmem, kTmemCols);
}

}  // namespace moda::d128

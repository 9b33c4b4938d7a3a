// MoDA backward, fused form: five contractions and one exponential per score.
//
// The paper prints no backward pass; this is the derivative of the Sec. 2.2 operator.  With
// P = exp(S - LSE) (sequence), R = exp(U - LSE) (depth), D_t = <dO_t, O_t>:
//
//   dS = P o (dO V^T - D),   dU_i = R_i (<dO, Vd_i> - D)
//   dQ = scale (dS K + sum_i dU_i Kd_i)     dK = scale dS^T Q     dV = P^T dO
//   dKd_i = scale dU_i Q                    dVd_i = R_i dO        (row-local)
//
// Four launches on the caller's stream:
//   0. bwd_prep_kernel        D_t, and a cleared fp32 dQ accumulator in the workspace.
//   1. bwd_rows_kernel        (l > 0) the depth part, local to a query row: for every depth slot R_i, dU_i, dKd_i, dVd_i
//                             (written in cache layout), and the row's depth share of dQ, added to the accumulator.
//                             Streams the depth cache exactly once, on a share of the SMs while 2. has the others.
//   2. moda_bwd_fused_kernel  one CTA per 128-key tile, looping over the 128-query tiles at or below the
//                             diagonal.  Per pair of tiles: S^T = K Q^T and dP^T = V dO^T (tcgen05, operands
//                             in shared memory; one extra k-step each adds the per-query terms -LSE / scale and
//                             -D_t to every score of the query's column), P^T and dS^T formed once by the row warps, dV += P^T dO (P^T
//                             from tensor memory), dK += dS^T Q and dQ_tile = dS K (dS^T staged once in shared
//                             memory and used by both: K-major for dK, MN-major for dQ).  dK, dV accumulate in
//                             tensor memory over the whole loop; the dQ tile is added to the fp32 accumulator
//                             in L2 by bulk reductions (cp.reduce.async.bulk .add.f32) from a staging buffer --
//                             the only place where the order of floating-point additions depends on scheduling.
//   3. bwd_dq_finish_kernel   dQ = bf16(scale * accumulator).
//
// Against the split form (moda_bwd.cuh: a dQ pass and a dK/dV pass, seven contractions, every score
// exponentiated twice, bit-reproducible) this form does 5/7 of the tensor work and half of the
// exponentials; the host picks it unless the caller asks for reproducible bits.
#pragma once

#include "moda_bwd.cuh"
#include "moda_cache.cuh"
#include "moda_fwd.cuh"
#include "moda_fwd_wide.cuh"
#include "sm100_ptx.cuh"

namespace moda {

// fp32 dQ accumulator: [b][h][query tile][feature / 4][row 128][4], so that a warp whose lanes own
// consecutive rows adds (or stores) 512 contiguous bytes per instruction.
inline size_t dq_acc_bytes(int B, int T, int H, int d) {
    return size_t(B) * H * num_tiles(T) * kTileRows * d * 4;
}
// Workspace of the fused backward: row terms D_t, then the dQ accumulator (256-byte aligned).
inline size_t bwd_fused_rowterm_bytes(int B, int T, int H) {
    return (size_t(B) * H * T * 4 + 255) & ~size_t(255);
}
inline size_t bwd_fused_workspace_bytes(int B, int T, int H, int d) {
    return bwd_fused_rowterm_bytes(B, T, H) + dq_acc_bytes(B, T, H, d);
}

// =====================================================================================
// 1. Row terms D_t = <dO_t, O_t>, and a cleared dQ accumulator
// =====================================================================================
// One CTA per (b, h, 128-row tile); D / 32 threads per row, each owning 32 features.  Bound by HBM: O and dO in, the
// fp32 accumulator out.
template <int D>
__global__ void __launch_bounds__(kTileRows * (D / 32))
bwd_prep_kernel(const __nv_bfloat16* __restrict__ O, const __nv_bfloat16* __restrict__ dO, float* __restrict__ delta,
                float* __restrict__ dq_acc, int B, int T, int H) {
    grid_launch_dependents();
    constexpr int PARTS = D / 32;                 // threads per row
    constexpr int CH = D / 8;                     // 16-byte chunks per row
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = lane % PARTS;
    const int r = warp * (32 / PARTS) + lane / PARTS;
    const int nq = num_tiles(T);
    const int qt = blockIdx.x % nq;
    const int bh = blockIdx.x / nq;
    const int b = bh / H, h = bh % H;
    const int t = qt * kTileRows + r;
    float dpart = 0.f;
    if (t < T) {
        const size_t row = ((size_t(b) * T + t) * H + h) * CH + part * 4;
        const uint4* o = reinterpret_cast<const uint4*>(O) + row;
        const uint4* g = reinterpret_cast<const uint4*>(dO) + row;
#pragma unroll
        for (int j = 0; j < 4; ++j) dpart += dot8_bf16(o[j], g[j]);
    }
#pragma unroll
    for (int off = 1; off < PARTS; off <<= 1) dpart += __shfl_xor_sync(0xffffffffu, dpart, off);
    if (t < T && part == 0) delta[(size_t(b) * H + h) * T + t] = dpart;
    float4* dst = reinterpret_cast<float4*>(dq_acc) + size_t(blockIdx.x) * (D / 4) * kTileRows + threadIdx.x;
#pragma unroll
    for (int j = 0; j < 8; ++j) dst[j * (kTileRows * PARTS)] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// =====================================================================================
// 3. dQ = bf16(scale * accumulator)
// =====================================================================================
// The launches of a backward overlap at their ends (programmatic dependent launch): this kernel, and a sequence part without
// a depth part before it, come up while the grid in front of them finishes and wait for it before they touch D_t or the accumulator.  Whole
// backward, graph replays, us, T = 100, l = 0, d = 64, 2 heads: 13.0 -> 10.9; 2 x 512, 16 heads, d = 128, l = 0: 24.0 -> 22.7; 2 x 1000, l = 0:
// 55.2 -> 54.1; T = 2000, 16 heads on 4, d = 64, l = 12: 119.3 -> 116.2; T = 1000, 8 heads, l = 7, e4m3 33.0 -> 32.6; from T = 4096 on nothing.  The
// sequence part lets this kernel start at the END of its CTAs: from their start on, its CTAs filled the few SMs that
// had no work in the last wave and did theirs there, four to an SM (2 x 1000, l = 0: 59.8; T = 512: 29.5).  So it is with the few SMs that the
// depth part leaves where that one ends last: with more CTAs here than such SMs they are let go behind it (B = 4, 32 heads, d = 128: T = 100, l = 64
// 189.3 -> 184.3, T = 128, l = 48 152.6 -> 148.2, T = 100, l = 6 35.8 -> 35.3); with fewer, beside it (2 x 100, 16 heads, d = 64, l = 3: 14.2, behind it 14.5).
template <int D>
__global__ void __launch_bounds__(kTileRows * (D / 32))
bwd_dq_finish_kernel(const float* __restrict__ dq_acc, __nv_bfloat16* __restrict__ dQ, int B, int T, int H, float scale) {
    constexpr int PARTS = D / 32;
    constexpr int CH = D / 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = lane % PARTS;
    const int r = warp * (32 / PARTS) + lane / PARTS;
    const int nq = num_tiles(T);
    const int qt = blockIdx.x % nq;
    const int bh = blockIdx.x / nq;
    const int b = bh / H, h = bh % H;
    const int t = qt * kTileRows + r;
    grid_dependency_wait();                       // started beside the end of the sequence part
    if (t >= T) return;
    const float4* src = reinterpret_cast<const float4*>(dq_acc) + size_t(blockIdx.x) * (D / 4) * kTileRows + size_t(part * 8) * kTileRows + r;
    uint4* dst = reinterpret_cast<uint4*>(dQ) + ((size_t(b) * T + t) * H + h) * CH + part * 4;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float4 a = __ldcs(src + (2 * j) * kTileRows);
        const float4 c = __ldcs(src + (2 * j + 1) * kTileRows);
        uint4 o;
        o.x = pack_bf16x2(a.x * scale, a.y * scale); o.y = pack_bf16x2(a.z * scale, a.w * scale);
        o.z = pack_bf16x2(c.x * scale, c.y * scale); o.w = pack_bf16x2(c.z * scale, c.w * scale);
        dst[j] = o;
    }
}

// =====================================================================================
// 2a. Row-local depth part: depth gradients and the depth share of dQ
// =====================================================================================
// A persistent grid of a share of the SMs (the host chooses it so that both parts end together).  It lets the next grid of
// the stream, the sequence part, start at once: this part moves every byte of the depth cache and of its gradient cache
// once and is bound by HBM, the sequence part by the tensor cores and L2, so one after the other leaves each resource idle
// in turn.  Both only add to the dQ accumulator; the sequence grid ends after this one has.
// Whole backward, ms, short runs, one after the other -> side by side: T = 4096, l = 23, d = 128, B = 4: 2.11 -> 1.66; T = 8192,
// l = 16, B = 2: 2.53 -> 2.15, e4m3 2.39 -> 2.01; T = 5000, l = 23, e4m3: 1.42 -> 1.11; T = 32768, l = 32, d = 64, 32 heads:
// 17.8 -> 16.6, e4m3 17.0 -> 15.9.
//
// A CTA walks units of 128 rows (d = 128; two tiles of 128 rows at d = 64, whose blocks are neighbours in the cache).
// Per unit the ring brings the Q and dO rows (TMA, 64 KiB) and then, slot by slot, the unit's K and V blocks (one
// contiguous run of the cache: 64 KiB in bf16, 33-34 KiB in e4m3).  A stage is released as soon as its bytes are in
// registers, so nearly the whole ring is in flight all the time.  D / 32 threads per row, each owning 32 features;
// lanes of a quarter warp own consecutive rows of one feature part: 128 contiguous bytes per access in the stage and
// in the gradient cache.  The two dot products of a slot are finished with shuffles; their terms are mixed-precision FMAs
// (unpacking the bf16 factors first made the arithmetic the bound: 2.7 us per 64 KiB in, 64 KiB out and SM against 1.55;
// 1.05 without the stores, which are the bound now).  With e4m3 codes they are packed fp32 FMAs, values before keys so that
// only the widened keys stay in registers: an entry takes 1.75 to 2.0 us as in bf16, against 2.2 (d = 128) and 2.7 (d = 64) with a
// scalar FMA per element.
struct RowsParams {
    const void* depth_kv;   // bf16 cache, or e4m3 codes + row scales (FP8 instantiation); gradients are bf16 either way
    __nv_bfloat16* d_depth_kv;
    const float *LSE, *delta;
    float* dq_acc;          // accumulator layout above; the depth share is added
    int B, T, H, l;
    int accumulate;         // nonzero: depth gradients are added to d_depth_kv (bf16 adds in L2)
    float scale, scale_log2;
};

template <int D, bool FP8>
struct RowsSmem {
    static constexpr int kTilesPerUnit = 128 / D;                        // 512 threads, 32 features each
    static constexpr int kQBytes = 4 * kTileRows * 128;                  // Q and dO rows of a unit: 64 KiB at either width
    static constexpr int kTileKV = FP8 ? 2 * (kTileRows * D + kTileRows * 4) : 2 * kTileRows * D * 2;   // K and V blocks of a tile
    static constexpr int kStages = 3;                                    // the Q, dO entry sets the stage size
    static constexpr int kStageBytes = 65536 + (FP8 ? 4096 : 0);
    static constexpr int kBars = kStages * kStageBytes;
    static constexpr int kMisc = kBars + 2 * kStages * 8;
    static constexpr int kTotal = kMisc + 16;
    static constexpr int kDynamic = kTotal + 1024;
    static_assert(kDynamic > 233472 / 2, "one CTA per SM: the sequence part beside it needs whole SMs too");
    static_assert(kTilesPerUnit * kTileKV <= kStageBytes && kQBytes <= kStageBytes, "a ring stage holds either kind of entry");
};

template <int D, bool FP8 = false>
__global__ void __launch_bounds__(512, 1)
bwd_rows_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapdO, const RowsParams p) {
    using R = RowsSmem<D, FP8>;
    constexpr int PARTS = D / 32, TPU = R::kTilesPerUnit, NSUB = D / 64;
    constexpr int RW = 32 / PARTS;                     // rows per warp
    constexpr int CH = D / 8;
    grid_launch_dependents();                          // the sequence part may take the SMs that this grid leaves
    if (g_moda_status != 0) return;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = aligned_dynamic_smem(smem_raw, R::kTotal);
    if (smem == nullptr) {
        if (threadIdx.x == 0) atomicCAS(&g_moda_status, 0, kStatusSmemLayout);
        return;
    }
    const uint32_t sbase = smem_u32(smem);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + R::kMisc);
    const int B = p.B, T = p.T, H = p.H, row_ctas = gridDim.x;
    const int tid = threadIdx.x, lane = tid & 31;
    const int hf = (TPU == 2) ? tid >> 8 : 0;          // which tile of the unit
    const int part = lane / RW;
    const int r = ((tid >> 5) & (4 * PARTS - 1)) * RW + lane % RW;
    const int nq = num_tiles(T);
    const int tiles = B * H * nq;
    const int units = (tiles + TPU - 1) / TPU;
    const int cta = blockIdx.x;
    const int my_units = (units - cta + row_ctas - 1) / row_ctas;
    const int n_total = my_units * (p.l + 1);          // ring entries: per unit one of Q, dO and l of K, V
    if (tid == 0) {
        *abort_flag = 0;
        for (int s = 0; s < R::kStages; ++s) {
            mbar_init(sbase + R::kBars + 8 * s, 1);
            mbar_init(sbase + R::kBars + 8 * (R::kStages + s), 16);
        }
        fence_mbar_init();
    }
    __syncthreads();
    const size_t slot_bytes = FP8 ? cache8_slot_bytes(B, T, H, D) : cache_slot_elems(B, T, H, D) * 2;
    const uint64_t policy = l2_policy_evict_first();
    // entry (unit index u, slot i; i = -1: Q and dO) into stage st
    auto issue = [&](int u, int i, int st) {
        const int first = (cta + u * row_ctas) * TPU;
        const int cnt = (TPU == 1 || first + 1 < tiles) ? TPU : 1;
        const uint32_t full = sbase + R::kBars + 8 * st, dst = sbase + st * R::kStageBytes;
        if (i < 0) {
            mbar_arrive_expect_tx(full, uint32_t(cnt) * (2 * kTileRows * D * 2));
            for (int k = 0; k < cnt; ++k) {
                const int bh = (first + k) / nq, qt = (first + k) % nq;
#pragma unroll
                for (int s = 0; s < NSUB; ++s) {
                    tma_load_4d(dst + k * (kTileRows * D * 4) + s * (kTileRows * 128), &mapQ, full, s * 64, bh % H, qt * kTileRows, bh / H);
                    tma_load_4d(dst + k * (kTileRows * D * 4) + (NSUB + s) * (kTileRows * 128), &mapdO, full, s * 64, bh % H, qt * kTileRows, bh / H);
                }
            }
        } else {
            const uint32_t bytes = uint32_t(cnt) * R::kTileKV;
            mbar_arrive_expect_tx(full, bytes);
            bulk_load(dst, static_cast<const uint8_t*>(p.depth_kv) + size_t(i) * slot_bytes + size_t(first) * R::kTileKV, bytes, full, policy);
        }
    };
    int iu = 0, ii = -1;                               // next entry to issue (thread 0)
    if (tid == 0) {
        tma_prefetch_desc(&mapQ);
        tma_prefetch_desc(&mapdO);
        for (int n = 0; n < R::kStages && n < n_total; ++n) {
            issue(iu, ii, n);
            if (++ii == p.l) { ii = -1; ++iu; }
        }
    }
    // row terms of the thread's row in unit u; rows past T: R = 0, zero gradients
    auto row_terms = [&](int u, float& neg_lse2, float& delta) {
        const int lt = (cta + u * row_ctas) * TPU + hf;
        neg_lse2 = -INFINITY;
        delta = 0.f;
        if (u < my_units && lt < tiles) {
            const int t = (lt % nq) * kTileRows + r;
            if (t < T) {
                const size_t idx = size_t(lt / nq) * T + t;
                neg_lse2 = -p.LSE[idx] * kLog2e;
                delta = p.delta[idx];
            }
        }
    };
    const size_t grad_stride = cache_slot_elems(B, T, H, D) / 8;         // slot of the gradient cache, in uint4
    const bool accumulate = p.accumulate != 0;
    float next_lse, next_delta;
    row_terms(0, next_lse, next_delta);
    int st = 0, phase = 0;
#pragma unroll 1
    for (int u = 0; u < my_units; ++u) {
        const int lt = (cta + u * row_ctas) * TPU + hf;
        const bool have = TPU == 1 || lt < tiles;      // the last unit of an odd number of tiles has one tile
        const float neg_lse2 = next_lse, delta = next_delta;
        row_terms(u + 1, next_lse, next_delta);
        uint4* gK = reinterpret_cast<uint4*>(p.d_depth_kv) + (size_t(lt) * 2 * CH + part * 4) * kTileRows + r;
        uint4 q4[4], g4[4];
        float acc[32];
#pragma unroll 1
        for (int i = -1; i < p.l; ++i) {
            const uint32_t full = sbase + R::kBars + 8 * st, empty = sbase + R::kBars + 8 * (R::kStages + st);
            const uint8_t* stage = smem + st * R::kStageBytes;
            mbar_wait(full, phase, abort_flag, 150);
            if (i < 0) {
                const uint8_t* qs = stage + hf * (kTileRows * D * 4);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    q4[j] = *reinterpret_cast<const uint4*>(qs + swz_chunk_offset(r, part * 4 + j));
                    g4[j] = *reinterpret_cast<const uint4*>(qs + kTileRows * D * 2 + swz_chunk_offset(r, part * 4 + j));
                }
                fence_proxy_async_smem();              // the refill (async proxy) comes after these loads
                __syncwarp();
                if (lane == 0) mbar_arrive(empty);
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[e] = 0.f;
            } else {
                float u_s = 0.f, dr = 0.f;
                float kf[FP8 ? 32 : 1];
                uint4 kc[FP8 ? 1 : 4];
                float sk = 1.f;
                if constexpr (FP8) {
                    const uint8_t* ks = stage + hf * R::kTileKV;
                    const uint8_t* vs = ks + kTileRows * D + kTileRows * 4;
                    uint4 k8[2], v8[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        k8[j] = *reinterpret_cast<const uint4*>(ks + ((part * 2 + j) * kTileRows + r) * 16);
                        v8[j] = *reinterpret_cast<const uint4*>(vs + ((part * 2 + j) * kTileRows + r) * 16);
                    }
                    sk = *reinterpret_cast<const float*>(ks + kTileRows * D + r * 4);
                    const float sv = *reinterpret_cast<const float*>(vs + kTileRows * D + r * 4);
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(empty);
                    // features 16 j + 4 k .. + 3 of this thread = halves of the packed q / dO words 2 (4 j + k), 2 (4 j + k) + 1; values
                    // first, so that only the widened keys (needed again for dQ) stay in registers
                    const uint32_t* qw = reinterpret_cast<const uint32_t*>(q4);
                    const uint32_t* gw = reinterpret_cast<const uint32_t*>(g4);
                    float u1 = 0.f, dr1 = 0.f;
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        float f0, f1, f2, f3;
                        e4m3x4_to_f32(reinterpret_cast<const uint32_t*>(v8)[m], f0, f1, f2, f3);
                        fma2_f32(bf16_lo_to_f32(gw[2 * m]), bf16_hi_to_f32(gw[2 * m]), f0, f1, dr, dr1);
                        fma2_f32(bf16_lo_to_f32(gw[2 * m + 1]), bf16_hi_to_f32(gw[2 * m + 1]), f2, f3, dr, dr1);
                    }
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        float* f = kf + 4 * m;
                        e4m3x4_to_f32(reinterpret_cast<const uint32_t*>(k8)[m], f[0], f[1], f[2], f[3]);
                        fma2_f32(bf16_lo_to_f32(qw[2 * m]), bf16_hi_to_f32(qw[2 * m]), f[0], f[1], u_s, u1);
                        fma2_f32(bf16_lo_to_f32(qw[2 * m + 1]), bf16_hi_to_f32(qw[2 * m + 1]), f[2], f[3], u_s, u1);
                    }
                    u_s += u1;
                    dr += dr1;
#pragma unroll
                    for (int off = RW; off < 32; off <<= 1) {
                        u_s += __shfl_xor_sync(0xffffffffu, u_s, off);
                        dr += __shfl_xor_sync(0xffffffffu, dr, off);
                    }
                    u_s *= sk;
                    dr *= sv;
                } else {
                    const uint4* ks = reinterpret_cast<const uint4*>(stage) + (hf * 2 * CH + part * 4) * kTileRows + r;
                    uint4 vc[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        kc[j] = ks[j * kTileRows];
                        vc[j] = ks[(CH + j) * kTileRows];
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(empty);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        u_s += dot8_bf16(q4[j], kc[j]);
                        dr += dot8_bf16(g4[j], vc[j]);
                    }
#pragma unroll
                    for (int off = RW; off < 32; off <<= 1) {
                        u_s += __shfl_xor_sync(0xffffffffu, u_s, off);
                        dr += __shfl_xor_sync(0xffffffffu, dr, off);
                    }
                }
                const float Rp = fast_exp2(fmaf(u_s, p.scale_log2, neg_lse2));       // the forward's LSE covers both key sets
                const float dU = Rp * (dr - delta);
                const uint32_t r2 = pack_bf16x2(Rp, Rp);
                const float sdu = dU * p.scale;
                const uint32_t sdu2 = pack_bf16x2(sdu, sdu);
                const float duk = dU * sk;                 // dQ share: dU * (scale_k * code)
                uint4* gV = gK + CH * kTileRows;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint4 ov, ok;
                    ov.x = mul_bf16x2(g4[j].x, r2); ov.y = mul_bf16x2(g4[j].y, r2);
                    ov.z = mul_bf16x2(g4[j].z, r2); ov.w = mul_bf16x2(g4[j].w, r2);
                    ok.x = mul_bf16x2(q4[j].x, sdu2); ok.y = mul_bf16x2(q4[j].y, sdu2);
                    ok.z = mul_bf16x2(q4[j].z, sdu2); ok.w = mul_bf16x2(q4[j].w, sdu2);
                    if (have) {
                        if (accumulate) {
                            red_add_bf16x2_v4(gV + j * kTileRows, ov);
                            red_add_bf16x2_v4(gK + j * kTileRows, ok);
                        } else {
                            __stcs(gV + j * kTileRows, ov);
                            __stcs(gK + j * kTileRows, ok);
                        }
                    }
                    if constexpr (FP8) {
#pragma unroll
                        for (int e = 0; e < 8; e += 2) fma2_f32(duk, duk, kf[8 * j + e], kf[8 * j + e + 1], acc[8 * j + e], acc[8 * j + e + 1]);
                    } else {
                        axpy_bf16x2(duk, kc[j].x, acc[8 * j + 0], acc[8 * j + 1]);
                        axpy_bf16x2(duk, kc[j].y, acc[8 * j + 2], acc[8 * j + 3]);
                        axpy_bf16x2(duk, kc[j].z, acc[8 * j + 4], acc[8 * j + 5]);
                        axpy_bf16x2(duk, kc[j].w, acc[8 * j + 6], acc[8 * j + 7]);
                    }
                }
                gK += grad_stride;
            }
            if (tid == 0 && iu < my_units) {
                mbar_wait(empty, phase, abort_flag, 151);
                issue(iu, ii, st);
                if (++ii == p.l) { ii = -1; ++iu; }
            }
            if (++st == R::kStages) { st = 0; phase ^= 1; }
        }
        if (have) {
            // the depth share of dQ (unscaled) joins the accumulator that the sequence part adds to
            float* dst = p.dq_acc + ((size_t(lt) * (D / 4) + part * 8) * kTileRows + r) * 4;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                red_add_f32_v4(dst + j * kTileRows * 4, acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
        }
    }
    __syncthreads();
    abort_teardown(abort_flag, 0);
    __syncthreads();
}

// =====================================================================================
// 2b. Sequence part: dK, dV and the dQ tiles
// =====================================================================================
// 512 threads (in warp order):
//   row warps    two warpgroups.  "Shared" (d = 128; d = 64 with few iterations a CTA): both work on the same iteration, a thread owns
//                one key row (= tensor-memory lane) and 64 of its 128 query columns.  "Alternate" (d = 64): they take alternate
//                iterations, a thread owns one key row and all 128 query columns.  Either way P^T, then dS^T.
//   drain warps  one warpgroup: a thread owns one query row of the dQ tile; it copies the row out of tensor memory
//                (which frees the region at once) and hands it, 8 KiB at a time through a staging ring in shared
//                memory, to bulk reductions into the fp32 accumulator, at whatever pace L2 takes them, without
//                holding up the row warps.
//   then         a loader warp (TMA tiles; the per-query terms as bf16 parts for the extra k-step) and three warps
//                that issue the contractions: S; dP (alternate: and dV); dV, dQ, dK (alternate: dK, dQ).  MMAs of
//                different warps are ordered by mbarriers only.  (One warp for all five, in the order in which they become
//                ready, took 1.5 times as long at d = 64: its waits and commits come one after the other.)
//
// Tensor memory (fp32 columns): X, 128 columns per buffer, S^T overlaid by P^T (bf16) -- one buffer at d = 128,
// two at d = 64 (where dK and dV leave room);  Y, 128 columns, dP^T;  dK, D columns;  dV, D columns.  512 columns at either head
// width.  The dQ tile takes Y behind dP^T of the same iteration (shared), or the half of an X buffer that P^T has left
// (alternate: dQ_i behind P_{i+1}, so that neither dP_{i+1} nor S_{i+1} waits for the copy).
//
// What bounds it (cycle stamps per warp role, T = 8192): the rate at which a dQ tile's additions are taken by L2 (64 KiB
// of fp32 per iteration per SM at d = 128; all SMs together sustain about 5.9 TB/s in a kernel that does nothing else,
// 4.3 TB/s here beside as many bytes of Q / dO loads): the drain warps need ~4300 cycles per tile, the five contractions
// 2700 tensor cycles.  The shared-memory port (MMA operands 304 KiB per iteration, TMA writes 64 KiB, dS^T 32 KiB, the
// dQ staging 64 KiB in and out, against 128 bytes per clock) is at two thirds of its peak since the row warps no
// longer load the per-query terms.
//
// Two dependency chains per shared iteration i, which overlap each other and the next iteration:
//   X:  S'_i = S_i - LSE / scale -> P_i^T = exp2(S' c) (row warps) -> dV_i -> X free -> S_{i+1}
//   Y:  dP'_i = dP_i - D -> dS_i^T = P o dP' to shared memory (row warps) -> dQ_i -> copied out (drain warps) -> Y free -> dP_{i+1}
// and dK_i, issued behind dQ_i, fills the tensor pipe while the row warps exponentiate tile i+1.
//
// At d = 64 the row warps set the pace: with both warpgroups on one iteration they exponentiate together (1320 cycles, the
// SFU's 1024 and latencies) and then form dS together (900, the SFU idle), 2650 cycles an iteration against some 1700 of the
// tensor cores (an SS MMA of N = 64 takes 48 cycles, its operands at 128 bytes a clock, not 32).  On alternate iterations
// one's exponentials overlap the other's dS.  What that needs: P^T in registers for a whole row (160 registers),
// dP_{i+1} as soon as dP_i is in registers, a second dS buffer, a fourth Q stage (a tile is in use for two and a half iterations
// and takes some 1200 cycles to arrive) -- paid for with two of the four staging chunks.  Cycles per iteration about 2300 now; T = 32768,
// 32 heads, whole backward 13.1 -> 11.3 ms (1.15-1.18), T = 16384, 64 heads on 8 6.8 -> 5.8, T = 8192, 16 heads 474 -> 425 us.
// With few iterations a CTA it loses (one warpgroup has the whole pass of an odd last one): bwd_alternates in launch_rules.h.  Measured on the way, T = 32768, gain over
// the shared iteration: scores in four loads of 32 columns, each waited for, 1.02 (all 128 requested at once: 1.15); dQ in its own tile's X
// buffer 1.07; dQ before dK 1.06; three Q stages and four chunks 1.04; chunks of 4 KiB 0.93, or of one warp's 32 rows (no barrier among
// the drain warps) 0.93; one X buffer with P^T and dQ in columns of their own 1.15.  dS^T in tensor memory as well, as dK's A operand,
// with the shared iteration: 1.01 (d = 128: 0.97).

// ALT: the two row warpgroups take alternate iterations; else both work on each, half of the query columns a warpgroup.
template <int D, bool ALT = (D == 64)>
struct FusedSmem {
    static_assert(!ALT || D == 64, "tensor memory has room for two S^T buffers at d = 64 only");
    static constexpr int kRowWGs = 2;                          // row warpgroups
    static constexpr int kThreads = (kRowWGs * 4 + 8) * 32;    // row warps, 4 drain warps, loader + 3 issuers
    static constexpr int kTileBytes = kTileRows * D * 2;       // 128 x D bf16
    static constexpr int kSubBytes = kTileRows * 128;          // 128 x 64 sub-tile (128-byte rows)
    // Stages of Q_i.  Q_i is read by S_i early and by dK_i late in its iteration, and a tile takes 1200 to 1600
    // cycles from the TMA issue to the first MMA that uses it, so with two stages the chain "dK_{i-2} completes ->
    // load Q_i -> S_i -> P_i -> dS_i -> dK_i" spans two iterations and sets the pace; alternate iterations, which are in flight for longer,
    // take four.
    static constexpr int kStages = (D == 128) ? 2 : ALT ? 4 : 3;
    // dO_i is read by dP_i and dV_i, both of which complete before dP_{i+1} can be issued; at d = 128 one
    // stage leaves the 32 KiB that the dQ staging buffer needs
    static constexpr int kdOStages = (D == 128) ? 1 : 2;
    static constexpr int kK = 0;
    static constexpr int kV = kK + kTileBytes;
    static constexpr int kQ = kV + kTileBytes;                 // stages of Q_i
    static constexpr int kdO = kQ + kStages * kTileBytes;      // stages of dO_i
    static constexpr int kdS = kdO + kdOStages * kTileBytes;   // dS^T: 128 keys x 128 queries bf16, one buffer per warpgroup that fills one
    static constexpr int kdSBytes = kTileRows * kTileRows * 2;
    static constexpr int kdSBufs = ALT ? 2 : 1;
    static constexpr int kStg = kdS + kdSBufs * kdSBytes;   // ring of 8 KiB chunks (16 feature columns of a dQ tile, fp32, accumulator layout)
    static constexpr int kStgSlots = (D == 128) ? 3 : ALT ? 2 : 4;       // d = 128: three as fast as four, two cost 3-4 %
    static constexpr int kStgBytes = kStgSlots * 16 * kTileRows * 4;
    // Operands of the extra k-step that adds the per-query terms to the two score contractions (see the kernel):
    // 2 KiB chunks of [128 rows][8 bf16] (unswizzled core matrices, 16 bytes per row): one per Q stage with the
    // stage's terms, then the two constant "ones" chunks and a zero chunk.
    static constexpr int kAug = kStg + kStgBytes;
    static constexpr int kAugChunk = kTileRows * 16;
    static constexpr int kAugOnesS = kAug + kStages * kAugChunk;
    static constexpr int kAugOnesD = kAugOnesS + kAugChunk;
    static constexpr int kAugZero = kAugOnesD + kAugChunk;
    static constexpr int kBars = kAugZero + kAugChunk;
    static constexpr int kNumBars = 32;
    static constexpr int kMisc = kBars + kNumBars * 8;
    static constexpr int kTotal = kMisc + 16;
    static constexpr int kSmemLimit = 232448;                  // 227 KiB per CTA on sm_100
    // the tiles need a 1024-byte aligned base; ask for the slack when it fits (d = 64), else rely on the
    // dynamic segment starting aligned and check at run time (aligned_dynamic_smem)
    static constexpr int kDynamic = (kTotal + 1024 <= kSmemLimit) ? kTotal + 1024 : kSmemLimit;
    static_assert(kTotal <= kSmemLimit, "shared-memory plan too large");
};

enum FusedBar : int {
    kFBarKV = 0,
    kFBarQFull = 1,     // +stage (<= 4), count 32: Q_i and the per-query terms of the stage have landed
    kFBarQEmpty = 5,    // +stage (<= 4): dK_i complete (Q_i, the row terms and, shared iterations, the dS buffer are free)
    kFBardOFull = 9,    // +stage (<= 2)
    kFBardOEmpty = 11,  // +stage (<= 2), count 2: dP_i and dV_i complete
    kFBarSFull = 13,    // +X buffer: S_i complete
    kFBarPFull = 15,    // +X buffer, count kRowArrivals: P_i^T written
    kFBardPFull = 17,   // +dS buffer: dP_i complete
    kFBardSFull = 19,   // +dS buffer, count kRowArrivals: dS_i^T written to shared memory, dP_i consumed
    kFBardSFree = 21,   // +dS buffer: dQ_i and dK_i complete (alternating warpgroups)
    kFBarXFree = 23,    // +X buffer: dV_i complete (alternating warpgroups: and dQ_i copied out): the buffer may take S_{i + buffers}
    kFBardQFull = 25,   // +dS buffer: dQ_i complete
    kFBarYFree = 27,    // count 128: dQ_i copied out (alternating warpgroups: dP_i in registers): Y may take dP_{i+1}
    kFBarFinal = 28,    // last dV and dK complete, count = warps that issue them
    kFBarDrain = 29,    // +issuer (3): abort path only
};

struct FusedParams {
    const float* LSE;
    const float* delta;
    float* dq_acc;
    int B, T, H;        // H = number of query heads
    int G;              // query heads per key/value head; dK, dV sum over the G heads of a group
    float scale, scale_log2;
    const uint4* slot_grad;     // SLOT: the slot of a gradient cache that dK, dV take up
    int beside_rows;    // launched beside bwd_rows_kernel (which has not finished): the grid must not end before it
    int finish_behind_rows;     // the finish kernel is let go behind that kernel as well
};

template <int D, bool SLOT = false, bool ALT = (D == 64)>
__global__ void __launch_bounds__(FusedSmem<D, ALT>::kThreads, 1)
moda_bwd_fused_kernel(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV,
                      const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapdO,
                      const __grid_constant__ CUtensorMap mapdK, const __grid_constant__ CUtensorMap mapdV,
                      const FusedParams p) {
    using L = FusedSmem<D, ALT>;
    constexpr int NSUB = D / 64;
    constexpr int NRW = L::kRowWGs, NROW = 128 * NRW;             // row warpgroups, row threads
    constexpr int kRowArrivals = ALT ? 128 : NROW;
    constexpr int W_DRAIN = 4 * NRW, W_LOAD = W_DRAIN + 4, W_S = W_LOAD + 1, W_DP = W_LOAD + 2;
    constexpr int W_ACC = W_LOAD + 3;                             // issues the three accumulating contractions
    constexpr int NOTHER = (L::kThreads / 32 - W_LOAD) * 32;      // threads of the loader / issuer warps
    constexpr uint32_t kTmemCols = 512;
    // d = 64 leaves room for a second S^T / P^T buffer: one per row warpgroup, or S_{i+1} while they work on tile i (B = 8, 32 heads, l = 0: T = 640
    // 128 us with one buffer, 124 with two; T = 256 42.5, 41.9)
    constexpr int XB = (D == 64) ? 2 : 1, WB = ALT ? 2 : 1;       // S^T / P^T buffers; dP, dS and dQ barriers
    constexpr uint32_t kColX = 0, kColY = 128 * XB, kColdK = kColY + 128, kColdV = kColdK + D;
    static_assert(kColdV + D <= kTmemCols, "tensor-memory plan too large");

    const bool last_cta = p.beside_rows && blockIdx.x == gridDim.x - 1;   // ends the grid after the rows kernel, on every path
    if (g_moda_status != 0) {
        grid_dependency_wait();
        return;
    }

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = aligned_dynamic_smem(smem_raw, L::kTotal);
    if (smem == nullptr) {
        if (threadIdx.x == 0) atomicCAS(&g_moda_status, 0, kStatusSmemLayout);
        grid_dependency_wait();
        return;
    }
    const uint32_t sbase = smem_u32(smem);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kMisc + 4);
    auto bar = [&](int i) { return sbase + L::kBars + 8u * uint32_t(i); };

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nk = num_tiles(p.T);
    const int bh = blockIdx.x / nk;
    const int kt = blockIdx.x % nk;                       // key tiles in ascending order: most work first
    const int Hk = p.H / p.G;
    const int b = bh / Hk, h = bh % Hk;                   // h: key/value head of this CTA
    const int k0 = kt * kTileRows;
    const int n_per = nk - kt;                            // query tiles kt .. nk-1 see this key tile
    const int n_it = n_per * p.G;                         // iteration it: query head h G + it / n_per, tile kt + it % n_per

    if (tid == 0) {
        *abort_flag = 0;
        mbar_init(bar(kFBarKV), 1);
        for (int s = 0; s < L::kStages; ++s) {
            mbar_init(bar(kFBarQFull + s), 32);
            mbar_init(bar(kFBarQEmpty + s), 1);
        }
        for (int s = 0; s < L::kdOStages; ++s) {
            mbar_init(bar(kFBardOFull + s), 1);
            mbar_init(bar(kFBardOEmpty + s), 2);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar(kFBarSFull + s), 1);
            mbar_init(bar(kFBarPFull + s), kRowArrivals);
            mbar_init(bar(kFBarXFree + s), ALT ? 129 : 1);
            mbar_init(bar(kFBardPFull + s), 1);
            mbar_init(bar(kFBardSFull + s), kRowArrivals);
            mbar_init(bar(kFBardSFree + s), 1);
            mbar_init(bar(kFBardQFull + s), 1);
        }
        mbar_init(bar(kFBarYFree), 128);
        mbar_init(bar(kFBarFinal), ALT ? 2 : 1);
        for (int s = 0; s < 3; ++s) mbar_init(bar(kFBarDrain + s), 1);
        fence_mbar_init();
    }
    if (warp == W_S) {
        tmem_alloc(smem_u32(tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    {   // constant chunks of the extra k-step: 1.0 in columns 0-2 (S) / 4-6 (dP), zero elsewhere; the per-stage chunks start
        // at zero because the chunk behind the one in use is read too (against the zero chunk: it only has to be finite)
        constexpr uint32_t kOne2 = 0x3F803F80u, kOne1 = 0x00003F80u;
        uint4* aug = reinterpret_cast<uint4*>(smem + L::kAug);
        for (int i = threadIdx.x; i < (L::kStages + 3) * kTileRows; i += L::kThreads) {
            const int chunk = i / kTileRows;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (chunk == L::kStages) v = make_uint4(kOne2, kOne1, 0u, 0u);
            if (chunk == L::kStages + 1) v = make_uint4(0u, 0u, kOne2, kOne1);
            aug[i] = v;
        }
        fence_proxy_async_smem();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    // Abort path of an issuing thread: wait (bounded) until its own MMAs have drained.
    auto drain_on_abort = [&](int which) {
        if (*abort_flag != 0) {
            umma_commit(bar(kFBarDrain + which));
            const uint64_t t0 = globaltimer_ns();
            while (!mbar_try_wait(bar(kFBarDrain + which), 0) && globaltimer_ns() - t0 < 20000000ull) {}
        }
    };

    // Register budget: the CTA owns what it was launched with (512 threads x 128 registers), and setmaxnreg.inc blocks until the CTA's own pool can serve it, so the three shares must fit that total.
    constexpr int kRegsLaunch = 128;
    static_assert(L::kThreads == 512, "the register shares below assume 512 threads");
    // Shares measured (T = 8192 .. 65536): the issuing warps need about 100 registers to keep their descriptors and
    // barrier addresses without spills; d = 128: 128 / 160 / 96 (42.1 ms at T = 65536 against 44.1 with 136 / 160 / 80).  Alternate iterations:
    // 128 scores and what becomes of them in a row thread, a dQ row of 64 in a drain thread; d = 64, shared: 28.5 ms with 152 / 152 / 56, 27.6 with
    // 136 / 136 / 104 (T = 32768, H = 32).
    constexpr int kRegsRow = (D == 128) ? 128 : ALT ? 160 : 136, kRegsDrain = (D == 128) ? 160 : ALT ? 96 : 136, kRegsOther = (D == 128 || ALT) ? 96 : 104;
    static_assert(NROW * kRegsRow + 128 * kRegsDrain + NOTHER * kRegsOther <= L::kThreads * kRegsLaunch, "register shares exceed the CTA's pool");
    // setmaxnreg.inc to less than the current count (or .dec to more) is an illegal instruction
    static_assert(kRegsRow >= kRegsLaunch && kRegsOther <= kRegsLaunch, "setmaxnreg direction");
    if (warp < W_DRAIN) {
        // =========================== row warps: P^T, dS^T, dK / dV epilogue ===========================
        setmaxnreg_inc<kRegsRow>();
        const int hc = warp >> 2;                            // which row warpgroup
        const int r = tid & 127;                             // key row inside the tile = TMEM lane
        const uint32_t lane_addr = uint32_t((warp & 3) * 32) << 16;
        if constexpr (ALT) {
            // this warpgroup's iterations: hc, hc + 2, ...  One key row and all 128 query columns of each.
            const uint32_t tXw = tmem + lane_addr + kColX + hc * 128, tYw = tmem + lane_addr + kColY;
            uint8_t* dsw = smem + L::kdS + hc * L::kdSBytes + r * 128;
            int qi = kt + hc, ph = 0;
#pragma unroll 1
            for (int it = hc; it < n_it; it += 2, qi += 2, ph ^= 1) {
                while (qi >= nk) qi -= n_per;
                uint32_t pk[64];                             // P_i^T of this thread: 128 values, bf16 pairs
                // ---- P_i^T ----
                mbar_wait(bar(kFBarSFull + hc), ph, abort_flag, 121);
                tc_fence_after_sync();
                {
                    uint32_t sv[4][32];
#pragma unroll
                    for (int c = 0; c < 4; ++c) tmem_ld32(tXw + c * 32, sv[c]);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint32_t(&pc)[16] = *reinterpret_cast<uint32_t(*)[16]>(pk + 16 * c);
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            // the contraction has already subtracted LSE / scale from every score of the query's column
                            float e0, e1;
                            mul2_f32(__uint_as_float(sv[c][2 * j]), __uint_as_float(sv[c][2 * j + 1]), p.scale_log2, p.scale_log2, e0, e1);
                            pc[j] = pack_bf16x2(fast_exp2(e0), fast_exp2(e1));
                        }
                    }
                    if (qi == kt) {                          // the query tile is the key tile itself: column j sees key row r iff j >= r
#pragma unroll
                        for (int j = 0; j < 64; ++j) {
                            if (2 * j < r) pk[j] &= 0xffff0000u;
                            if (2 * j + 1 < r) pk[j] &= 0x0000ffffu;
                        }
                    }
                    tmem_st32(tXw, *reinterpret_cast<uint32_t(*)[32]>(pk));     // overlays columns that this thread has read
                    tmem_st32(tXw + 32, *reinterpret_cast<uint32_t(*)[32]>(pk + 32));
                }
                tmem_wait_st();
                tc_fence_before_sync();
                mbar_arrive(bar(kFBarPFull + hc));

                // ---- dS_i^T = P o (dP - D), with the bf16 P that dV uses ----
                mbar_wait(bar(kFBardPFull + hc), ph, abort_flag, 122);
                tc_fence_after_sync();
                if (it >= 2) mbar_wait(bar(kFBardSFree + hc), ph ^ 1, abort_flag, 123);    // dQ_{i-2}, dK_{i-2} have read the buffer
                {
                    uint32_t gv[2][32];
                    tmem_ld32(tYw, gv[0]);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (c < 3) tmem_ld32(tYw + (c + 1) * 32, gv[(c + 1) & 1]);
                        const uint32_t(&y)[32] = gv[c & 1];
#pragma unroll
                        for (int g = 0; g < 4; ++g) {        // 8 query columns = one 16-byte chunk of the row
                            uint32_t w[4];                   // gv holds dP - D_t already (subtracted by the contraction)
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const uint32_t pp = pk[16 * c + 4 * g + k];
                                float x0, x1;
                                mul2_f32(bf16_lo_to_f32(pp), bf16_hi_to_f32(pp), __uint_as_float(y[8 * g + 2 * k]), __uint_as_float(y[8 * g + 2 * k + 1]), x0, x1);
                                w[k] = pack_bf16x2(x0, x1);
                            }
                            *reinterpret_cast<uint4*>(dsw + (c >> 1) * L::kSubBytes + ((((c & 1) * 4 + g) ^ (r & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                        }
                        if (c < 3) tmem_wait_ld();
                        if (c == 2) {
                            tc_fence_before_sync();
                            mbar_arrive(bar(kFBarYFree));    // dP_i is in registers: Y may take dP_{i+1}
                        }
                    }
                }
                fence_proxy_async_smem();                    // generic-proxy stores -> read by the MMAs (async proxy)
                tc_fence_before_sync();
                mbar_arrive(bar(kFBardSFull + hc));
            }
        } else {
        constexpr int COLS = kTileRows / NRW;                // query columns per thread, of every iteration
        static_assert(COLS == 64, "a 64-column sub-tile of dS^T per warpgroup");
        const uint32_t tX0 = tmem + lane_addr + kColX + hc * COLS, tY = tmem + lane_addr + kColY + hc * COLS;
        uint8_t* ds_row = smem + L::kdS + hc * L::kSubBytes + r * 128;
#pragma unroll 1
        for (int it = 0, qi = kt; it < n_it; ++it, qi = (qi + 1 < nk) ? qi + 1 : kt) {
            uint32_t pk[COLS / 2];                           // P_i^T of this thread: COLS values, bf16 pairs
            // ---- P_i^T ----
            const int xb = it % XB;
            const uint32_t tX = tX0 + xb * 128;
            mbar_wait(bar(kFBarSFull + xb), (it / XB) & 1, abort_flag, 121);
            tc_fence_after_sync();
            {
                // all blocks are requested before the first is used: the later loads' latency hides under the
                // first block's exponentials
                uint32_t sv[COLS];
#pragma unroll
                for (int c = 0; c < COLS / 32; ++c) tmem_ld32(tX + c * 32, *reinterpret_cast<uint32_t(*)[32]>(sv + c * 32));
                tmem_wait_ld();
#pragma unroll
                for (int i4 = 0; i4 < COLS / 4; ++i4) {
                    // the contraction has already subtracted LSE / scale from every score of the query's column (packed
                    // products, here and for dS^T: 64 instructions fewer per tile, the same bits; d = 64 1-2 % faster)
                    float e0, e1, e2, e3;
                    mul2_f32(__uint_as_float(sv[4 * i4 + 0]), __uint_as_float(sv[4 * i4 + 1]), p.scale_log2, p.scale_log2, e0, e1);
                    mul2_f32(__uint_as_float(sv[4 * i4 + 2]), __uint_as_float(sv[4 * i4 + 3]), p.scale_log2, p.scale_log2, e2, e3);
                    e0 = fast_exp2(e0);
                    e1 = fast_exp2(e1);
                    e2 = fast_exp2(e2);
                    e3 = fast_exp2(e3);
                    pk[2 * i4] = pack_bf16x2(e0, e1);
                    pk[2 * i4 + 1] = pack_bf16x2(e2, e3);
                }
            }
            if (qi == kt) {                                  // the query tile is the key tile itself: column c sees key row r iff c >= r
                const int first = r - hc * COLS;             // (masked here and not in the loop above: it stays off the path of every other tile)
#pragma unroll
                for (int j = 0; j < COLS / 2; ++j) {
                    if (2 * j < first) pk[j] &= 0xffff0000u;
                    if (2 * j + 1 < first) pk[j] &= 0x0000ffffu;
                }
            }
            // P^T (bf16, two per column) overlays the first half of the columns this thread has read
            tmem_st32(tX, pk);
            tmem_wait_st();
            tc_fence_before_sync();
            mbar_arrive(bar(kFBarPFull + xb));

            // ---- dS_i^T = P o (dP - D), with the bf16 P that dV uses ----
            mbar_wait(bar(kFBardPFull), it & 1, abort_flag, 122);
            tc_fence_after_sync();
            // the dS buffer is still read by dQ_{i-1} and dK_{i-1} (dK is issued last: its completion covers both)
            if (it > 0) mbar_wait(bar(kFBarQEmpty + (it - 1) % L::kStages), ((it - 1) / L::kStages) & 1, abort_flag, 123);
            {
                uint32_t gv[COLS];
#pragma unroll
                for (int c = 0; c < COLS / 32; ++c) tmem_ld32(tY + c * 32, *reinterpret_cast<uint32_t(*)[32]>(gv + c * 32));
                tmem_wait_ld();
#pragma unroll
                for (int g = 0; g < COLS / 8; ++g) {         // 8 query columns = one 16-byte chunk of the row
                    uint32_t w[4];                           // gv holds dP - D_t already (subtracted by the contraction)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        float x0, x1;
                        mul2_f32(bf16_lo_to_f32(pk[4 * g + k]), bf16_hi_to_f32(pk[4 * g + k]), __uint_as_float(gv[8 * g + 2 * k]),
                                 __uint_as_float(gv[8 * g + 2 * k + 1]), x0, x1);
                        w[k] = pack_bf16x2(x0, x1);
                    }
                    const uint4 v = make_uint4(w[0], w[1], w[2], w[3]);
                    *reinterpret_cast<uint4*>(ds_row + ((g ^ (r & 7)) << 4)) = v;
                }
            }
            fence_proxy_async_smem();                        // generic-proxy stores -> read by the MMAs (async proxy)
            tc_fence_before_sync();
            mbar_arrive(bar(kFBardSFull));
        }

        }
        // ---- epilogue: dK (scaled) by the first warpgroup, dV by the second ----
        // In a stack the later layers' gradient of this layer's K, V lies in a slot of the gradient cache, whose K or V block
        // of this tile is laid out as the threads read it here (chunk, then row: 512 contiguous bytes per warp).  A copy kernel
        // behind the backward would read and write dK, dV once more: 12.5 us a layer at 2 x 1000 positions of 16 heads, and the pass
        // of four layers and four projected slots took 798 us of device time with it, 767 without.  The loads run ahead of
        // their use.  An instantiation of its own: with the test at run time the backward without a slot was 0.7 % slower at T = 1000.
        const uint4* sg = p.slot_grad + (size_t(blockIdx.x) * 2 + hc) * (kTileRows * (D / 8)) + r;
        uint4 more[2][4] = {};
        const auto load_more = [&](int c) {
#pragma unroll
            for (int g = 0; g < 4; ++g)
                more[c & 1][g] = __ldcs(sg + (c * 4 + g) * kTileRows);
        };
        if constexpr (SLOT) load_more(0);
        mbar_wait(bar(kFBarFinal), 0, abort_flag, 124);
        tc_fence_after_sync();
        {
            const float mul = hc == 0 ? p.scale : 1.f;
            const uint32_t col = hc == 0 ? kColdK : kColdV;
            const int dst_off = hc == 0 ? L::kQ : L::kdO;    // every MMA has completed: the stages are free
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
                if (SLOT && c + 1 < D / 32) load_more(c + 1);
                uint32_t o[32];
                tmem_ld32(tmem + lane_addr + col + c * 32, o);
                tmem_wait_ld();
#pragma unroll
                for (int g4 = 0; g4 < 4; ++g4) {
                    uint4 v;
                    const uint4 m = more[c & 1][g4];
                    const auto sum = [&](int i, uint32_t w) {
                        const float x0 = __uint_as_float(o[8 * g4 + i]), x1 = __uint_as_float(o[8 * g4 + i + 1]);
                        if constexpr (!SLOT) return pack_bf16x2(x0 * mul, x1 * mul);
                        else return pack_bf16x2(fmaf(x0, mul, bf16_lo_to_f32(w)), fmaf(x1, mul, bf16_hi_to_f32(w)));
                    };
                    v.x = sum(0, m.x);
                    v.y = sum(2, m.y);
                    v.z = sum(4, m.z);
                    v.w = sum(6, m.w);
                    *reinterpret_cast<uint4*>(smem + dst_off + swz_chunk_offset(r, c * 4 + g4)) = v;
                }
            }
        }
        fence_proxy_async_smem();
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (tid == 0) {
#pragma unroll
            for (int s = 0; s < NSUB; ++s) {
                tma_store_4d(&mapdK, sbase + L::kQ + s * L::kSubBytes, s * 64, h, k0, b);
                tma_store_4d(&mapdV, sbase + L::kdO + s * L::kSubBytes, s * 64, h, k0, b);
            }
            tma_store_commit();
            tma_store_wait_read();
        }
    } else if (warp < W_LOAD) {
        // =========================== drain warps: dQ tile -> fp32 accumulator ===========================
        // The tile leaves the SM as bulk reductions (cp.reduce.async.bulk, fp32 add in L2) from a staging buffer
        // in shared memory.  Per-thread red.global instructions would do the same additions, but they queue in the
        // load/store path of the SM at the pace L2 takes them, and every shared-memory load, store and barrier probe of
        // the row warps then waits behind them (measured: + 2000 cycles per iteration).
        if constexpr (kRegsDrain >= kRegsLaunch) setmaxnreg_inc<kRegsDrain>();
        else setmaxnreg_dec<kRegsDrain>();
        const int r = tid & 127;                             // query row inside the tile = TMEM lane
        const uint32_t tdQ = tmem + (uint32_t((warp & 3) * 32) << 16) + (ALT ? kColX + 64 : kColY);
        if (ALT) mbar_arrive(bar(kFBarXFree));               // no dQ tile lies in the first S^T buffer's other half yet
        float4* stg = reinterpret_cast<float4*>(smem + L::kStg) + r;          // [feature / 4 (16)][row 128] float4
        float* dst = p.dq_acc + ((size_t(b) * p.H + h * p.G) * nk + kt) * (size_t(kTileRows) * D);
        int slot = 0;
#pragma unroll 1
        for (int it = 0, qi = kt; it < n_it; ++it) {
            const int xb = it % WB;
            mbar_wait(bar(kFBardQFull + xb), (it / WB) & 1, abort_flag, 120);
            tc_fence_after_sync();
            uint32_t o[D];
#pragma unroll
            for (int c = 0; c < D / 32; ++c) tmem_ld32(tdQ + (ALT ? (xb ^ 1) * 128 : 0) + c * 32, *reinterpret_cast<uint32_t(*)[32]>(o + c * 32));
            tmem_wait_ld();
            tc_fence_before_sync();
            mbar_arrive(bar(ALT ? kFBarXFree + (xb ^ 1) : kFBarYFree));   // X may take S of the iteration after the next / Y may take dP of the next
            // 16 feature columns (8 KiB, contiguous in the accumulator) at a time through a ring of staging chunks:
            // a chunk is rewritten once the reduction issued from it one ring earlier has finished reading it, so
            // all but one of the ring's reductions stay in flight and L2, not this loop, sets the pace.
#pragma unroll
            for (int ch = 0; ch < D / 16; ++ch) {
                if (tid == NROW) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(L::kStgSlots - 1) : "memory");
                asm volatile("bar.sync 2, 128;" ::: "memory");
#pragma unroll
                for (int g = 0; g < 4; ++g)
                    stg[(slot * 4 + g) * kTileRows] = make_float4(__uint_as_float(o[ch * 16 + 4 * g]), __uint_as_float(o[ch * 16 + 4 * g + 1]),
                                                                  __uint_as_float(o[ch * 16 + 4 * g + 2]), __uint_as_float(o[ch * 16 + 4 * g + 3]));
                fence_proxy_async_smem();
                asm volatile("bar.sync 2, 128;" ::: "memory");
                if (tid == NROW) {
                    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;"
                                 ::"l"(dst + ch * (16 * kTileRows)), "r"(sbase + L::kStg + slot * (16 * kTileRows * 4)), "r"(16 * kTileRows * 4) : "memory");
                    tma_store_commit();
                }
                slot = (slot + 1 == L::kStgSlots) ? 0 : slot + 1;          // the ring runs on across iterations
            }
            dst += kTileRows * D;
            if (++qi == nk) {                                // the next query head of the group
                qi = kt;
                dst += size_t(kt) * (kTileRows * D);
            }
        }
        if (tid == NROW) tma_store_wait_all();               // the finish kernel may be up already: the sums are in place
    } else {
      setmaxnreg_dec<kRegsOther>();
      constexpr uint32_t idesc_acc = make_idesc_bf16(128, D, false, true);
      const uint64_t dvb0 = desc_mnmajor_sw128(sbase + L::kdO, 0, L::kSubBytes);
      // dV += P^T dO (P^T from tensor memory, dO MN-major); dst = stage of dO_i, xb = X buffer of P_i
      auto issue_dV = [&](int it, int dst, int xb) {
          const uint64_t dvb = dvb0 + uint64_t((dst * L::kTileBytes) >> 4);
          // 16 queries per k-step: 8 columns; with half the columns per row warpgroup, in the block of the one that owns them
#pragma unroll 4
          for (int kk = 0; kk < kTileRows / 16; ++kk)
              umma_ts(tmem + kColdV, tmem + kColX + xb * 128 + (ALT ? kk * 8 : (kk >> 2) * 64 + (kk & 3) * 8), dvb + uint64_t(kk * 128),
                      idesc_acc, (it > 0 || kk > 0) ? 1u : 0u);
          umma_commit(bar(kFBarXFree + xb));
          umma_commit(bar(kFBardOEmpty + dst));
      };
      if (warp == W_LOAD) {
        // =========================== loader: TMA tiles + per-query LSE, D_t ===========================
        if (lane == 0) {
            tma_prefetch_desc(&mapK);
            tma_prefetch_desc(&mapV);
            tma_prefetch_desc(&mapQ);
            tma_prefetch_desc(&mapdO);
            mbar_arrive_expect_tx(bar(kFBarKV), 2 * L::kTileBytes);
#pragma unroll
            for (int s = 0; s < NSUB; ++s) {
                tma_load_4d(sbase + L::kK + s * L::kSubBytes, &mapK, bar(kFBarKV), s * 64, h, k0, b);
                tma_load_4d(sbase + L::kV + s * L::kSubBytes, &mapV, bar(kFBarKV), s * 64, h, k0, b);
            }
        }
        // without a depth part this grid starts beside the prep kernel, which writes D_t and clears the dQ accumulator
        if (!p.beside_rows) grid_dependency_wait();
        const float inv_scale = 1.f / p.scale;
        int hq = h * p.G, qrow0 = k0;
#pragma unroll 1
        for (int it = 0; it < n_it; ++it) {
            const int st = it % L::kStages;
            const size_t row_base = (size_t(b) * p.H + hq) * p.T;
            // lane handles query columns 4 lane .. 4 lane + 3: for each, -LSE / scale and -D_t as three bf16 parts
            // (hi + mid + lo = the fp32 value); queries past T get a large negative first term so that P = 0
            uint4 av[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = qrow0 + 4 * lane + j;
                const float nl = (c < p.T) ? -p.LSE[row_base + c] * inv_scale : -1.0e30f;
                const float nd = (c < p.T) ? -__ldcg(p.delta + row_base + c) : 0.f;
                av[j] = make_uint4(0u, 0u, 0u, 0u);
                split3_bf16(nl, av[j].x, av[j].y);
                split3_bf16(nd, av[j].z, av[j].w);
            }
            if (it >= L::kStages) mbar_wait(bar(kFBarQEmpty + st), ((it - L::kStages) / L::kStages) & 1, abort_flag, 130);
            uint4* aug = reinterpret_cast<uint4*>(smem + L::kAug + st * L::kAugChunk) + 4 * lane;
#pragma unroll
            for (int j = 0; j < 4; ++j) aug[j] = av[j];
            fence_proxy_async_smem();                        // generic-proxy stores -> read by the MMAs (async proxy)
            if (lane == 0) {
                mbar_arrive_expect_tx(bar(kFBarQFull + st), L::kTileBytes);
#pragma unroll
                for (int s = 0; s < NSUB; ++s)
                    tma_load_4d(sbase + L::kQ + st * L::kTileBytes + s * L::kSubBytes, &mapQ, bar(kFBarQFull + st), s * 64, hq, qrow0, b);
                const int dst = it % L::kdOStages;
                if (it >= L::kdOStages) mbar_wait(bar(kFBardOEmpty + dst), ((it - L::kdOStages) / L::kdOStages) & 1, abort_flag, 131);
                mbar_arrive_expect_tx(bar(kFBardOFull + dst), L::kTileBytes);
#pragma unroll
                for (int s = 0; s < NSUB; ++s)
                    tma_load_4d(sbase + L::kdO + dst * L::kTileBytes + s * L::kSubBytes, &mapdO, bar(kFBardOFull + dst), s * 64, hq, qrow0, b);
            } else {
                mbar_arrive(bar(kFBarQFull + st));
            }
            qrow0 += kTileRows;
            if (qrow0 >= nk * kTileRows) {                   // the next query head of the group
                qrow0 = k0;
                ++hq;
            }
        }
      } else if (warp == W_S || warp == W_DP) {
        // ============ MMA issuers: S^T = K Q^T (warp 13, into X), dP^T = V dO^T (warp 14, into Y) ============
        {   // whole warp: operands are warp-uniform, one elected lane issues
            const bool is_s = (warp == W_S);
            constexpr uint32_t idesc_s = make_idesc_bf16(128, 128, false, false);
            const uint32_t a_tile = sbase + (is_s ? L::kK : L::kV);
            const int full0 = is_s ? kFBarQFull : kFBardOFull;
            const int nb = is_s ? XB : 1;                                 // accumulator buffers of this contraction
            // a descriptor of a later k-step is the first one plus a compile-time constant (the start-address field
            // counts 16-byte units and stays inside its 14 bits below 256 KiB)
            const uint64_t da0 = desc_kmajor_sw128(a_tile, 0);
            const uint64_t db0 = desc_kmajor_sw128(sbase + (is_s ? L::kQ : L::kdO), 0);
            // extra k-step: A = ones in the columns of this contraction's terms (second k-chunk: the zero chunk),
            // B = the Q stage's chunk of per-query terms (second k-chunk: whatever follows it, finite, times zero)
            const uint64_t da_aug = make_smem_desc_noswz(sbase + (is_s ? L::kAugOnesS : L::kAugOnesD),
                                                         uint32_t(L::kAugZero - (is_s ? L::kAugOnesS : L::kAugOnesD)), 128u);
            const uint64_t db_aug0 = make_smem_desc_noswz(sbase + L::kAug, uint32_t(L::kAugChunk), 128u);
            mbar_wait(bar(kFBarKV), 0, abort_flag, 140);
            const int nst = is_s ? L::kStages : L::kdOStages;
#pragma unroll 1
            for (int it = 0; it < n_it; ++it) {
                const int st = it % nst;
                // the accumulator buffer still holds P of its previous tile (until that dV completes) / dQ_{i-1} (until
                // it is copied out)
                const int xb = it % nb;
                const uint32_t col = is_s ? kColX + xb * 128 : kColY;
                const uint32_t free_bar = is_s ? bar(kFBarXFree + xb) : bar(kFBarYFree);
                const int ob = it % WB;
                if (it >= nb) mbar_wait2(bar(full0 + st), (it / nst) & 1, free_bar, ((it - nb) / nb) & 1, abort_flag, 141, is_s ? 142 : 143);
                else mbar_wait(bar(full0 + st), (it / nst) & 1, abort_flag, 141);
                // dP also needs the Q stage's per-query terms (they arrive with Q_i)
                const int qst = it % L::kStages;
                if (!is_s) mbar_wait(bar(kFBarQFull + qst), (it / L::kStages) & 1, abort_flag, 147);
                tc_fence_after_sync();
                const uint64_t db = db0 + uint64_t((st * L::kTileBytes) >> 4);
#pragma unroll 1
                for (int c = 0; c < NSUB; ++c) {
                    const uint64_t ca = da0 + uint64_t(c * (L::kSubBytes >> 4)), cb = db + uint64_t(c * (L::kSubBytes >> 4));
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) umma_ss(tmem + col, ca + uint64_t(kk * 2), cb + uint64_t(kk * 2), idesc_s, (c > 0 || kk > 0) ? 1u : 0u);
                }
                umma_ss(tmem + col, da_aug, db_aug0 + uint64_t((qst * L::kAugChunk) >> 4), idesc_s, 1u);
                umma_commit(bar(is_s ? kFBarSFull + xb : kFBardPFull + ob));
                if (!is_s) umma_commit(bar(kFBardOEmpty + st));
                // P_i is written before dP_i is consumed, so dV_i never holds up dP_{i+1}
                if (ALT && !is_s) {
                    mbar_wait(bar(kFBarPFull + ob), (it / XB) & 1, abort_flag, 144);
                    tc_fence_after_sync();
                    issue_dV(it, st, ob);
                }
            }
            if (ALT && !is_s) umma_commit(bar(kFBarFinal));
            drain_on_abort(is_s ? 0 : 1);
        }
      } else if (warp == W_ACC) {
        // ============ MMA issuer of the accumulating contractions.  Shared iterations: dV_i += P^T dO (P^T from tensor memory, dO MN-major),
        // ============ then, once dS_i^T is in shared memory, dQ_tile = dS K into Y (dS^T and K both MN-major) and
        // ============ dK += dS^T Q (dS^T K-major, Q MN-major).  P_i, dS_i, P_{i+1} are produced in this order, so one
        // ============ warp can take the three in turn.  dQ before dK: its tile has to be copied out before dP of the next
        // ============ iteration can land, dK only has to finish before dS_{i+1} is written.  Alternate: dK_i, then dQ_i, whose columns
        // ============ P_{i+1} has to leave first.
        {
            constexpr uint32_t idesc_dq = make_idesc_bf16(128, D, true, true);
            const uint64_t dqa0 = desc_mnmajor_sw128(sbase + L::kdS, 0, L::kSubBytes);
            const uint64_t dqb0 = desc_mnmajor_sw128(sbase + L::kK, 0, L::kSubBytes);
            const uint64_t dka0 = desc_kmajor_sw128(sbase + L::kdS, 0);
            const uint64_t dkb0 = desc_mnmajor_sw128(sbase + L::kQ, 0, L::kSubBytes);
#pragma unroll 1
            for (int it = 0; it < n_it; ++it) {
                const int st = it % L::kStages, dst = it % L::kdOStages, xb = it % XB, wb = it % WB;
                if constexpr (!ALT) {
                    mbar_wait2(bar(kFBarPFull + xb), (it / XB) & 1, bar(kFBardOFull + dst), (it / L::kdOStages) & 1, abort_flag, 144, 145);
                    tc_fence_after_sync();
                    issue_dV(it, dst, xb);
                }
                const uint64_t dsb = uint64_t((wb * L::kdSBytes) >> 4);
                mbar_wait(bar(kFBardSFull + wb), (it / WB) & 1, abort_flag, 146);
                tc_fence_after_sync();
                const uint64_t dkb = dkb0 + uint64_t((st * L::kTileBytes) >> 4);
                auto issue_dK = [&]() {
#pragma unroll 4
                    for (int kk = 0; kk < kTileRows / 16; ++kk)
                        umma_ss(tmem + kColdK, dka0 + dsb + uint64_t(((kk >> 2) * L::kSubBytes + (kk & 3) * 32) >> 4), dkb + uint64_t(kk * 128),
                                idesc_acc, (it > 0 || kk > 0) ? 1u : 0u);
                    umma_commit(bar(kFBarQEmpty + st));
                };
                if constexpr (ALT) {
                    // dK first: dQ_i goes to the half of the other X buffer that P_{i+1} leaves (the last tile: whose dQ tile has been copied out)
                    issue_dK();
                    if (it + 1 < n_it) mbar_wait(bar(kFBarPFull + (xb ^ 1)), ((it + 1) / XB) & 1, abort_flag, 148);
                    else if (it > 0) mbar_wait(bar(kFBarXFree + (xb ^ 1)), ((it - 1) / XB) & 1, abort_flag, 149);
                    tc_fence_after_sync();
                }
#pragma unroll 4
                for (int kk = 0; kk < kTileRows / 16; ++kk)
                    umma_ss(tmem + (ALT ? kColX + (xb ^ 1) * 128 + 64 : kColY), dqa0 + dsb + uint64_t(kk * 128), dqb0 + uint64_t(kk * 128), idesc_dq, kk > 0);
                umma_commit(bar(kFBardQFull + wb));
                if constexpr (ALT) umma_commit(bar(kFBardSFree + xb));
                else issue_dK();
            }
            umma_commit(bar(kFBarFinal));
            drain_on_abort(2);
        }
      }
    }

    tc_fence_before_sync();
    __syncthreads();
    abort_teardown(abort_flag, 256);
    __syncthreads();
    // the finish kernel may come up: beside the end of the rows kernel if there is room for it on the SMs that one leaves
    if (last_cta && p.finish_behind_rows) grid_dependency_wait();
    grid_launch_dependents();
    if (warp == W_S) tmem_dealloc(tmem, kTmemCols);
    // what follows on the stream reads the accumulator and the depth gradients: this grid ends after the rows kernel has
    if (last_cta) grid_dependency_wait();
}

}  // namespace moda

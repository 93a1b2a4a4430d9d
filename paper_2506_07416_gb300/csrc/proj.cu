// Layer-0 projection that makes the queries and keys the scores read (Design
// section: the module is the first decoder layer, whose q and k are
// RoPE(W . RMSNorm(x))):
//     s_r    = 1 / sqrt(mean_h x_r[h]^2 + eps)
//     y_r[o] = s_r * sum_h x_r[h] * W'[o][h] + bias[o],   W' = W * gamma (per input column)
// then rotary position embedding per head (rotate-half pairs j, j + d/2) with
// cos / sin from a table indexed by the row's position.
//
// The RMSNorm weight is folded into W once (fold kernel below), so the
// contraction reads the raw hidden rows; the per-row scale s_r is a sum of
// squares taken from the A tiles while they sit in shared memory for the tensor
// core, and is applied in the epilogue with the bias and the rotation.
//
// Pairs of CTAs (clusters of two, cta_group::2) work through output tiles of 256
// rows x BN columns (BN = 256, or 128 where the columns leave no choice), N tiles
// fastest, so that the tiles in flight share their rows of x and W' stays in L2.
// Each CTA stages its 128 rows of x and half of the tile's rows of W' (64 hidden
// values a stage); warp 1 of the first CTA issues the tcgen05.mma (M = 256,
// N = BN, K = 16) for both, so a CTA's operands take 64 bytes a clock out of shared
// memory and 64 in (one CTA alone on 128 x 256: 96 and 96; its limit is 128).
// Accumulators alternate between two TMEM buffers: the epilogue of a tile runs
// under the contraction of the next.
//   warp 0: TMA producer; warp 1: TMEM, and in the first CTA the MMA issuer; warps
//   6-9: row sums, each stage after its contraction and before it is given back;
//   warps 2-5: epilogue (TMEM lane = row); warps 6-9 take half of a pair's last
//   tile, after which there is nothing left to sum.
// Against one-CTA tiles of 256 x 256 with a single accumulator, whose sums shared
// the tile's stages with the contraction: 27648 x 4096 -> 4096 755 -> 617 us, 6157
// x 3584 -> 512 (e4m3) 34.3 -> 26.6 us, 1536 x 2048 -> 2048 25.5 -> 19.4 us (48 tiles
// on 76 pairs: 10 us of it are launch, set-up and the one epilogue); with the
// contractions issued from uniform registers (elect_one) 588, 24.9 and 18.5 us, and
// with stages held until their sums have their values and the closing exchange about
// waits that gave up 603, 25.2 and 18.8. A
// kernel of its own for the row scales, overlapping the first tiles, was slower on
// all of them (623, 29 and 21 us against 617, 26.6 and 19.4): its loads compete with
// the copies.
// Every wait is bounded. When one gives up the pair brings its copies level and waits
// for the barriers of all that it started before it leaves.

#include <math.h>

#include <cuda_fp8.h>

#include "internal.h"
#include "pipe.cuh"
#include "ptx.cuh"

namespace lvs {

namespace {

constexpr int kProjThreads = 320;  // producer, MMA issuer, epilogue warpgroup, summing warpgroup
constexpr int kProjK = 64;         // hidden values per stage (128 bytes of bf16)
constexpr int kProjRows = 128;     // rows of a tile per CTA

template <int BN>
struct ProjLayout {
    static constexpr int A_BYTES = kProjRows * 128;
    static constexpr int B_BYTES = BN / 2 * 128;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int STAGES = 192 * 1024 / STAGE;
    static constexpr int OFF_A = 0;
    static constexpr int OFF_B = OFF_A + STAGES * A_BYTES;
    static constexpr int OFF_ROPE = OFF_B + STAGES * B_BYTES;  // 4 KB per epilogue warp
    // full[S], done[S], empty[S], acc_full[2], acc_empty[2], sc_full[2], sc_empty[2], drain, stall
    static constexpr int OFF_BAR = OFF_ROPE + 8 * 4096;
    static constexpr int OFF_SC = OFF_BAR + (3 * STAGES + 10) * 8;  // [2][128] row scales
    static constexpr int OFF_MISC = OFF_SC + 2 * kProjRows * 4;
    // TMEM address, abort flag, the other CTA's; ProjCounts of this CTA and of the other
    static constexpr int OFF_COUNTS = OFF_MISC + 16;
    static constexpr int ALLOC = OFF_COUNTS + 2 * 16 + 1024;
    static constexpr int TMEM_COLS = 2 * BN;
};

// What a CTA of a pair had started when its roles ended: stages it copied, and (first
// CTA) stages contracted and accumulators committed.
struct ProjCounts {
    int copied, contracted, tiles, unused;
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// The rotation of a pair: y1 cos - y2 sin and y2 cos + y1 sin, with the product by
// the cosine fused into the sum. Spelled out: which product the compiler fuses
// changed with the code around it, and with it one output in 100,000 by one bf16 step.
__device__ __forceinline__ float rotate_lo(float y1, float y2, float c, float s)
{
    return __fmaf_rn(y1, c, -__fmul_rn(y2, s));
}
__device__ __forceinline__ float rotate_hi(float y1, float y2, float c, float s)
{
    return __fmaf_rn(y2, c, __fmul_rn(y1, s));
}

// two e4m3 codes (round to nearest even, saturating to +-448)
__device__ __forceinline__ uint32_t pack_e4m3(float lo, float hi)
{
    return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, __NV_E4M3);
}

// 2 * NP consecutive outputs of one row from NP value pairs: bf16, or e4m3 codes
// of y / scale when the call asked for e4m3
template <int NP>
__device__ __forceinline__ void store_pairs(const ProjArgs& p, int64_t elem, const float2 (&y)[NP])
{
    if (p.y8) {
        uint32_t o[NP / 2];
#pragma unroll
        for (int q = 0; q < NP / 2; ++q)
            o[q] = pack_e4m3(y[2 * q].x * p.out_inv_scale, y[2 * q].y * p.out_inv_scale) |
                   (pack_e4m3(y[2 * q + 1].x * p.out_inv_scale, y[2 * q + 1].y * p.out_inv_scale) << 16);
        uint4* d = reinterpret_cast<uint4*>(p.y8 + elem);
#pragma unroll
        for (int q = 0; q < NP / 8; ++q) d[q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
    } else {
        uint32_t o[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) o[q] = pack_bf16(y[q].x, y[q].y);
        uint4* d = reinterpret_cast<uint4*>(p.y + elem);
#pragma unroll
        for (int q = 0; q < NP / 4; ++q) d[q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
    }
}

// A warp's window on the rotation table: the (cos, sin) pairs [16 c, 16 c + 16) of
// its 32 rows' positions, 128 bytes a row, in 4 KB of its own shared memory. The
// warp fetches four rows per load instruction (eight lanes a row, whole 128-byte
// lines); lane r then reads row r, whose 16-byte pieces are stored at piece ^ (r &
// 7) so that eight lanes hit eight different bank groups. A lane reading its own
// row straight from global memory touches 32 lines per instruction: 5 M of an L1's
// wavefronts on 6912 x 4096 -> 4096, 28 instead of 18 us on 1536 x 2048 -> 2048.
struct RopeWindow {
    const float2* table;
    uint8_t* buf;
    int half, pos, lane;
    uint4 next[8];

    __device__ __forceinline__ void fetch(int c)
    {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int rp = __shfl_sync(0xffffffffu, pos, 4 * i + (lane >> 3));
            const float2* src = table + (int64_t)rp * half + 16 * c + 2 * (lane & 7);
            const float2 a = __ldg(src), b = __ldg(src + 1);
            next[i] = make_uint4(__float_as_uint(a.x), __float_as_uint(a.y), __float_as_uint(b.x), __float_as_uint(b.y));
        }
    }
    __device__ __forceinline__ void put()
    {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = 4 * i + (lane >> 3);
            *reinterpret_cast<uint4*>(buf + r * 128 + (((lane & 7) ^ (r & 7)) << 4)) = next[i];
        }
        __syncwarp();
    }
    __device__ __forceinline__ float4 pairs(int j) const  // pairs 2j and 2j + 1 of this lane's row
    {
        return *reinterpret_cast<const float4*>(buf + lane * 128 + ((j ^ (lane & 7)) << 4));
    }
};

// scale, bias, rotation and store (bf16 or e4m3) of part `part` of `parts` of the BN
// columns of one accumulator row (this thread's): with a rotation, of every head's
// chunks of 16 pairs, the warp's window holding the part's first chunk in flight
// (fetched); without, of the columns.
template <int BN>
__device__ __forceinline__ void proj_store_row(const ProjArgs& p, uint32_t ta, int64_t grow, int n0, int part, int parts,
                                               bool live, float sc, RopeWindow& w)
{
    const int64_t row0 = grow * (int64_t)p.out_features + n0;  // element index of this tile's first column
    if (p.head_dim > 0) {
        const int half = p.head_dim / 2, nc = half / 16 / parts * (part + 1);
        for (int c = half / 16 / parts * part; c < nc; ++c) {
            w.put();
            if (c + 1 < nc) w.fetch(c + 1);
            for (int h0 = 0; h0 < BN; h0 += p.head_dim) {
                float v1[16], v2[16];
                tmem_ld16(ta + (uint32_t)(h0 + 16 * c), v1);
                tmem_ld16(ta + (uint32_t)(h0 + half + 16 * c), v2);
                tmem_wait_ld();
                const int col = n0 + h0 + 16 * c;
                float2 a[8], b[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 cs = w.pairs(j);
                    const float y1 = fmaf(v1[2 * j], sc, p.bias ? p.bias[col + 2 * j] : 0.f);
                    const float y2 = fmaf(v2[2 * j], sc, p.bias ? p.bias[col + half + 2 * j] : 0.f);
                    const float z1 = fmaf(v1[2 * j + 1], sc, p.bias ? p.bias[col + 2 * j + 1] : 0.f);
                    const float z2 = fmaf(v2[2 * j + 1], sc, p.bias ? p.bias[col + half + 2 * j + 1] : 0.f);
                    a[j] = make_float2(rotate_lo(y1, y2, cs.x, cs.y), rotate_lo(z1, z2, cs.z, cs.w));
                    b[j] = make_float2(rotate_hi(y1, y2, cs.x, cs.y), rotate_hi(z1, z2, cs.z, cs.w));
                }
                if (live) {
                    store_pairs(p, row0 + h0 + 16 * c, a);
                    store_pairs(p, row0 + h0 + half + 16 * c, b);
                }
            }
        }
    } else {
        for (int c = BN / parts * part; c < BN / parts * (part + 1); c += 32) {
            float v[32];
            tmem_ld32(ta + (uint32_t)c, v);
            tmem_wait_ld();
            if (live) {
                float2 o[16];
#pragma unroll
                for (int j = 0; j < 32; j += 2)
                    o[j / 2] = make_float2(fmaf(v[j], sc, p.bias ? p.bias[n0 + c + j] : 0.f),
                                           fmaf(v[j + 1], sc, p.bias ? p.bias[n0 + c + j + 1] : 0.f));
                store_pairs(p, row0 + c, o);
            }
        }
    }
}

template <int BN>
__global__ void __launch_bounds__(kProjThreads, 1)
    proj_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                const __grid_constant__ ProjArgs p)
{
    using L = ProjLayout<BN>;
    constexpr int S = L::STAGES;
    static_assert(L::ALLOC > 116 * 1024 && L::ALLOC <= 227 * 1024, "one CTA per SM");
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (base - raw);
    const int warp = uniform((int)(threadIdx.x >> 5)), lane = threadIdx.x & 31;
    const int rank = uniform((int)cluster_ctarank());
    const int pair = (int)(blockIdx.x >> 1), npairs = (int)(gridDim.x >> 1);
    const int nk = (p.hidden + kProjK - 1) / kProjK;
    const int ntn = p.out_features / BN;
    const int ntiles = (int)((p.rows + 2 * kProjRows - 1) / (2 * kProjRows)) * ntn;

    const uint32_t bar0 = base + L::OFF_BAR;
    auto FULL = [&](int s) -> uint32_t { return bar0 + 8u * (uint32_t)s; };
    auto DONE = [&](int s) -> uint32_t { return bar0 + 8u * (uint32_t)(S + s); };
    auto EMPTY = [&](int s) -> uint32_t { return bar0 + 8u * (uint32_t)(2 * S + s); };
    auto ACC_FULL = [&](int b) -> uint32_t { return bar0 + 8u * (uint32_t)(3 * S + b); };
    auto ACC_EMPTY = [&](int b) -> uint32_t { return bar0 + 8u * (uint32_t)(3 * S + 2 + b); };
    auto SC_FULL = [&](int b) -> uint32_t { return bar0 + 8u * (uint32_t)(3 * S + 4 + b); };
    auto SC_EMPTY = [&](int b) -> uint32_t { return bar0 + 8u * (uint32_t)(3 * S + 6 + b); };
    const uint32_t DRAIN = bar0 + 8u * (uint32_t)(3 * S + 8), STALL = DRAIN + 8u;
    float* sc_s = reinterpret_cast<float*>(smem + L::OFF_SC);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::OFF_MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::OFF_MISC + 4);
    volatile int* peer_abort = reinterpret_cast<volatile int*>(smem + L::OFF_MISC + 8);
    volatile ProjCounts* counts = reinterpret_cast<volatile ProjCounts*>(smem + L::OFF_COUNTS);

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(FULL(s), 1);   // first CTA: its arming arrival; both CTAs' copies complete bytes on it
            mbar_init(DONE(s), 1);   // the commit of the stage's contractions, in both CTAs
            mbar_init(EMPTY(s), 4);  // the summing warps
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(ACC_FULL(b), 1);
            mbar_init(ACC_EMPTY(b), 8);  // first CTA: the epilogue warps of both
            mbar_init(SC_FULL(b), 4);
            mbar_init(SC_EMPTY(b), 4);
        }
        mbar_init(DRAIN, 1);
        mbar_init(STALL, 1);  // nothing ever arrives (the debug stall below)
        *abort_flag = 0;
        *peer_abort = 0;
        counts[0].copied = counts[0].contracted = counts[0].tiles = 0;
        fence_mbar_init_cluster();
    }
    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&tm_x);
        tma_prefetch_desc(&tm_w);
    }
    if (warp == 1) {
        tmem_alloc_pair(smem_u32(tmem_slot), L::TMEM_COLS);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    cluster_sync_all();  // both CTAs' barriers and TMEM exist
    const uint32_t tmem = uniform(*tmem_slot);
    const Ctl ctl{abort_flag, p.err, p.wait_budget};
    volatile int no_abort = 0;
    const Ctl drain{&no_abort, p.err, kWaitBudgetCycles};
    griddep_wait();
    griddep_launch_dependents();

    // this CTA's first rows of x and W' of tile t, and the copies of the tile's stage kc
    // from there into slot s of the ring
    auto x_row = [&](int t) { return t / ntn * (2 * kProjRows) + rank * kProjRows; };
    auto w_row = [&](int t) { return t % ntn * BN + rank * (BN / 2); };
    auto load_stage = [&](int s, int kc, int m0, int n0) {
        const uint32_t full = mapa_shared(FULL(s), 0);
        if (rank == 0) mbar_arrive_expect_tx(FULL(s), 2u * (uint32_t)L::STAGE);
        tma_load_3d_pair(base + L::OFF_A + s * L::A_BYTES, &tm_x, full, kc * kProjK, 0, m0);
        tma_load_3d_pair(base + L::OFF_B + s * L::B_BYTES, &tm_w, full, kc * kProjK, 0, n0);
    };

    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            for (int t = pair; t < ntiles && ok; t += npairs) {
                const int m0 = x_row(t), n0 = w_row(t);
                for (int kc = 0; kc < nk; ++kc, ++it) {
                    const int s = it % S;
                    // Debug stall (p.stall, a test of the failure path): a pair's second CTA
                    // stops after three stages, so that the two give up with different counts
                    // of copies and of contractions in flight.
                    if (p.stall && rank == 1 && it == 3 && !wait_phase(STALL, 0, ctl)) { ok = false; break; }
                    if (!wait_phase(EMPTY(s), ((uint32_t)(it / S) & 1u) ^ 1u, ctl)) { ok = false; break; }
                    load_stage(s, kc, m0, n0);
                }
            }
            // every stage's last contraction has completed (and with it its copies),
            // its commit has arrived here and its rows are summed before this CTA leaves
            for (int s = 0; s < S && s < it && ok; ++s)
                ok = wait_phase(EMPTY(s), (uint32_t)((it - 1 - s) / S) & 1u, ctl);
            counts[0].copied = it;
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer (first CTA)
        if (rank == 0) {
            const uint32_t idesc = idesc_make(256, BN, 1u);
            int it = 0, a = 0, tiles = 0;
            bool ok = true;
            for (int t = pair; t < ntiles && ok; t += npairs, ++a) {
                const uint32_t d = tmem + (uint32_t)((a & 1) * BN);
                if (!__all_sync(0xffffffffu, wait_phase_cluster(ACC_EMPTY(a & 1), ((uint32_t)(a >> 1) & 1u) ^ 1u, ctl))) break;
                tc_fence_after();
                for (int kc = 0; kc < nk; ++kc, ++it) {
                    const int s = it % S;
                    if (!wait_phase_warp(FULL(s), (uint32_t)(it / S) & 1u, ctl)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t ad = sdesc_k_sw128(base + L::OFF_A + s * L::A_BYTES);
                    const uint64_t bd = sdesc_k_sw128(base + L::OFF_B + s * L::B_BYTES);
                    if (elect_one()) {
#pragma unroll
                        for (int st = 0; st < 4; ++st)
                            mma_f16_pair(d, ad + (uint64_t)st * 2, bd + (uint64_t)st * 2, idesc, (kc | st) != 0);
                        mma_commit_pair(DONE(s));
                    }
                    __syncwarp();
                }
                if (!ok) break;
                if (elect_one()) mma_commit_pair(ACC_FULL(a & 1));
                __syncwarp();
                ++tiles;
            }
            // Every contraction above has landed once this arrives. It arrives here alone:
            // nobody in the other CTA would wait for it before leaving.
            if (elect_one()) mma_commit_pair(DRAIN, 1);
            __syncwarp();
            wait_phase_warp(DRAIN, 0, drain);
            if (lane == 0) {
                counts[0].contracted = it;
                counts[0].tiles = tiles;
            }
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- row sums (wg 1), epilogue
        const int quad = warp & 3;
        const int wg = (warp - 2) >> 2;
        const int r = quad * 32 + lane;  // row of this CTA's half = TMEM lane
        RopeWindow w;
        w.table = p.rope;
        w.buf = smem + L::OFF_ROPE + (warp - 2) * 4096;
        w.half = p.head_dim / 2;
        w.lane = lane;
        // part `part` of `parts` of tile t, the a-th of this pair. A warp agrees on what
        // its waits found, here and below: a lane that gave up alone would leave the
        // others at their shuffles and aligned loads.
        auto store_tile = [&](int t, int a, int part, int parts) -> bool {
            const int64_t grow = (int64_t)(t / ntn) * (2 * kProjRows) + rank * kProjRows + r;
            if (p.head_dim > 0) {
                w.pos = grow < p.rows ? p.positions[grow] : 0;
                if (w.pos < 0 || w.pos >= p.max_positions) {
                    atomicOr(p.err, kErrBounds);
                    w.pos = 0;
                }
                w.fetch(w.half / 16 / parts * part);
            }
            if (!wait_phase_warp(SC_FULL(a & 1), (uint32_t)(a >> 1) & 1u, ctl)) return false;
            const float sc = sc_s[(a & 1) * kProjRows + r];
            __syncwarp();
            if (wg == 0 && lane == 0) mbar_arrive(SC_EMPTY(a & 1));
            if (!wait_phase_warp(ACC_FULL(a & 1), (uint32_t)(a >> 1) & 1u, ctl)) return false;
            tc_fence_after();
            proj_store_row<BN>(p, tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)((a & 1) * BN), grow, t % ntn * BN,
                               part, parts, grow < p.rows, sc, w);
            return true;
        };
        int it = 0, a = 0;
        bool ok = true;
        for (int t = pair; t < ntiles && ok; t += npairs, ++a) {
            const bool last = t + npairs >= ntiles;
            if (wg == 0) {
                if (!store_tile(t, a, 0, last ? 2 : 1)) break;
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_remote(mapa_shared(ACC_EMPTY(a & 1), 0));
                continue;
            }
            float2 ss = make_float2(0.f, 0.f);  // even and odd hidden values, each in order
            for (int kc = 0; kc < nk; ++kc, ++it) {
                const int s = it % S;
                if (!wait_phase_warp(DONE(s), (uint32_t)(it / S) & 1u, ctl)) { ok = false; break; }
                const uint8_t* row = smem + L::OFF_A + s * L::A_BYTES + r * 128;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint4 v = *reinterpret_cast<const uint4*>(row + ((j ^ (r & 7)) << 4));
                    const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 x = make_float2(__uint_as_float(w4[q] << 16), __uint_as_float(w4[q] & 0xFFFF0000u));
                        ss = ffma2(x, x, ss);
                    }
                }
                // Only this arrival keeps the next copy (async proxy) out of the stage
                // while the loads above (generic proxy) read it. An arrival orders no
                // proxies, and a load that has been issued but waits behind the stores of
                // the epilogue warps would read the copy's bytes. So every lane orders its
                // loads before the async proxy, and the arrival depends on a vote that
                // needs every lane's sums, hence the values of all its loads (a sum of
                // squares is never negative: the vote is always 0).
                fence_proxy_async_shared();
                const bool bad = __any_sync(0xffffffffu, ss.x < 0.f || ss.y < 0.f);
                if (lane == 0 && !bad) mbar_arrive(EMPTY(s));
            }
            if (!ok || !wait_phase_warp(SC_EMPTY(a & 1), ((uint32_t)(a >> 1) & 1u) ^ 1u, ctl)) break;
            sc_s[(a & 1) * kProjRows + r] = rsqrtf((ss.x + ss.y) / (float)p.hidden + p.eps);
            __syncwarp();
            if (lane == 0) mbar_arrive(SC_FULL(a & 1));
            if (last) store_tile(t, a, 1, 2);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) st_shared_cluster(mapa_shared(base + L::OFF_MISC + 8, rank ^ 1), 1);
    __syncwarp();
    cluster_sync_all();  // both CTAs are done with each other's barriers and contractions
    if (*abort_flag || *peer_abort) {
        // A wait gave up in one of them: copies may be under way and arrivals
        // outstanding that nobody waited for. The CTAs exchange what they started; the
        // contractions of the first have completed (DRAIN).
        const uint32_t to = mapa_shared(base + L::OFF_COUNTS + (uint32_t)sizeof(ProjCounts), rank ^ 1);
        if (threadIdx.x == 0) {
            st_shared_cluster(to, counts[0].copied);
            st_shared_cluster(to + 4, counts[0].contracted);
            st_shared_cluster(to + 8, counts[0].tiles);
        }
        __syncwarp();
        cluster_sync_all();
        if (threadIdx.x == 0) {
            // A slot's barrier completes a phase when both CTAs have copied into it. They
            // are at most a ring apart (a slot is refilled after a contraction over both),
            // so the one behind copies what it lacks, into slots that no contraction reads
            // any more. The phase before a slot's last was waited for when the slot was
            // refilled, so the last one's parity decides; the same holds for the commits.
            const int copied = max(counts[0].copied, counts[1].copied);
            for (int it = counts[0].copied; it < copied; ++it) {
                const int t = pair + it / nk * npairs;
                load_stage(it % S, it % nk, x_row(t), w_row(t));
            }
            if (rank == 0)
                for (int s = 0; s < S && s < copied; ++s) wait_phase(FULL(s), (uint32_t)((copied - 1 - s) / S) & 1u, drain);
            const int contracted = counts[rank].contracted, tiles = counts[rank].tiles;
            for (int s = 0; s < S && s < contracted; ++s)
                wait_phase(DONE(s), (uint32_t)((contracted - 1 - s) / S) & 1u, drain);
            for (int b = 0; b < 2 && b < tiles; ++b) wait_phase(ACC_FULL(b), (uint32_t)((tiles - 1 - b) / 2) & 1u, drain);
        }
        __syncwarp();
        cluster_sync_all();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, L::TMEM_COLS);
    }
}

// W'[o][h] = bf16(W[o][h] * gamma[h])
__global__ void fold_norm_kernel(const __nv_bfloat16* __restrict__ w, const float* __restrict__ gamma,
                                 __nv_bfloat16* __restrict__ out, int64_t total, int hidden)
{
    griddep_wait();
    griddep_launch_dependents();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = __float2bfloat16_rn(__bfloat162float(w[i]) * gamma[i % hidden]);
}

// table[p][j] = (cos, sin) of the fp32 angle p * inv_freq[j]
__global__ void rope_table_kernel(const RopeArgs a)
{
    griddep_wait();
    griddep_launch_dependents();
    const int64_t total = (int64_t)a.max_positions * a.half;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int pos = (int)(i / a.half), j = (int)(i % a.half);
        float s, c;
        sincosf((float)pos * a.inv_freq[j], &s, &c);
        a.table[i] = make_float2(c, s);
    }
}

template <class... Args>
cudaError_t launch_plain(void (*kern)(Args...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream,
                         Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <int BN>
cudaError_t launch_proj_variant(const CUtensorMap& tm_x, const CUtensorMap& tm_w, const ProjArgs& p, int num_sms,
                                cudaStream_t stream)
{
    using L = ProjLayout<BN>;
    auto kern = proj_kernel<BN>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::ALLOC);
    if (e != cudaSuccess) return e;
    const int64_t ntiles = (p.rows + 2 * kProjRows - 1) / (2 * kProjRows) * (p.out_features / BN);
    const int64_t pairs = ntiles < num_sms / 2 ? ntiles : num_sms / 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * pairs), 1, 1);
    cfg.blockDim = dim3(kProjThreads, 1, 1);
    cfg.dynamicSmemBytes = L::ALLOC;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = pdl_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, tm_x, tm_w, p);
}

}  // namespace

int proj_tile_cols(int out_features) { return out_features % 256 == 0 ? 256 : 128; }

cudaError_t launch_proj(const CUtensorMap& tm_x, const CUtensorMap& tm_w, const ProjArgs& p, int num_sms,
                        cudaStream_t stream)
{
    if (p.rows <= 0) return cudaSuccess;
    return proj_tile_cols(p.out_features) == 256 ? launch_proj_variant<256>(tm_x, tm_w, p, num_sms, stream)
                                                 : launch_proj_variant<128>(tm_x, tm_w, p, num_sms, stream);
}

cudaError_t launch_fold_norm(const __nv_bfloat16* w, const float* gamma, __nv_bfloat16* out, int64_t total,
                             int hidden, int num_sms, cudaStream_t stream)
{
    if (total <= 0) return cudaSuccess;
    const int64_t want = (total + 255) / 256;
    const unsigned grid = (unsigned)(want < 8LL * num_sms ? want : 8LL * num_sms);
    return launch_plain(fold_norm_kernel, grid, 256, 0, stream, w, gamma, out, total, hidden);
}

cudaError_t launch_rope_table(const RopeArgs& a, int num_sms, cudaStream_t stream)
{
    const int64_t total = (int64_t)a.max_positions * a.half;
    if (total <= 0) return cudaSuccess;
    const int64_t want = (total + 255) / 256;
    const unsigned grid = (unsigned)(want < 8LL * num_sms ? want : 8LL * num_sms);
    return launch_plain(rope_table_kernel, grid, 256, 0, stream, a);
}

}  // namespace lvs

// Visual-token importance scores on the sm_103a tensor cores.
//
// Computes, for every visual token j of request b (Design section, Token
// Selection Module: first-decoder-layer self-attention as importance, FastV
// style; scale 1/sqrt(d), softmax over the request's visual tokens, mean over
// query heads and text tokens):
//     score[j] = 1/(Hq*T) * sum_h sum_i exp(s_hij - m_hi) / l_hi
// without ever writing the logits s to memory.
//
// Work decomposition. One thread-block cluster of C CTAs serves one (request,
// head group); CTA r of the cluster owns a contiguous range of 128-token tiles
// of the request. For every query head h of the group:
//   pass 1: D1 = Q_h * K_tile^T on tcgen05 (M = 64 or 128 query rows, N = 128
//           visual columns) into TMEM; each epilogue thread keeps, for its text
//           row, a reference logit and the sum of 2^((s - ref) * c) over its
//           columns of the CTA's tiles;
//   exchange: each CTA publishes its per-row (ref, sum) in shared memory and
//           signals every CTA of the cluster by remote mbarrier arrivals; each
//           CTA merges the C partials in rank order (deterministic) into
//           b_hi = m_hi * c + log2(l_hi), c = scale * log2(e);
//   pass 2: D2 = K_tile * Q_h^T (M = 128 visual rows, N = T rounded up to 16)
//           into TMEM; one epilogue thread per visual token adds
//           sum_i 2^(s_ij * c - b_hi) to its running score.
// Text rows are packed: the hp query heads of one key head that fit beside each
// other in 128 rows (hp * T <= 128) form a head block, row i * hp + h of its Q
// tile being text row i of head h. "Head" below means such a block: it streams
// the key head's tiles once instead of hp times (last-token queries of 64
// requests, 32 / 8 heads: 282 -> 106 us; choose_score_kernel now gives that call to
// the resident kernel, 80).
// A CTA without a cluster works through several (request, head group) items,
// claimed largest first (in the no-alloc call, which shares nothing, there is a CTA
// per item): its set-up and teardown (5 us) are paid once, and the
// groups can be finer. Scores of 12 requests of 322 to 2491 tokens, 32 / 8 heads: 45
// -> 38 us; 16 requests of 636 to 2586, 16 heads: 36.5 -> 33.9; 32 requests of 629 to
// 3404 in e4m3, 32 heads: 109 -> 106.
// Software pipeline with one head of look-ahead: pass 1 of head s+1 runs while
// the statistics of head s travel across the cluster, then pass 2 of head s
// (a CTA that is its own cluster has nothing to wait for and runs the two
// passes of each head back to back).
// The K tiles stream through a TMA ring for both passes (the pass-2 re-read of
// a CTA's few tiles is normally served by L2). Scores are summed over the heads
// of the group in shared memory; with one head group they are final, with
// several the CTAs write partial rows and a small kernel launched behind this one
// adds them in a fixed order over all SMs (the last CTA of a request to finish
// used to: 28 rows of 1280 tokens through one SM made a tail of 6 to 8 us).
//
// The reference of pass 1 is not the running maximum: any logit near the row's
// largest serves, since the sums are floating point and the reference cancels in b.
// A thread takes the largest of the first 32 columns it sees, and moves it (to the
// larger maximum, rescaling its sum) only when a tile adds more than 2^12 to the sum,
// checked once per tile while the logits are still in tensor memory. So no exponent
// that counts is above 12, where its rounding (2^-21) is that of b, and the sum's
// logarithm stays about as small as under the maximum. (A limit of 2^96, which only
// keeps the sums finite, let errors of a row reach 3.8e-6; now 4.2e-7, and 5.4e-7 with
// the running maximum. Redone tiles cost the e4m3 item above 6% at 2^8, 1% at 2^10 and
// nothing at 2^12; the lower limits were no more exact on ordinary batches.) In units of
// log2 the reference is rounded to a whole number, so that sums under two references
// are merged by a power of two, without error. The loop is then one fused multiply-add
// (packed in pairs), one 2^x and one add (packed) per logit, in both passes.
//
// Warp roles (352 threads): warp 0 = TMA producer, warps 1 and 2 = MMA issuers
// (warp 1 also allocates TMEM), warps 3..10 = epilogue, two warpgroups (TMEM
// lane quadrant = warp % 4). A contraction unit is one tile of one pass; the
// units cycle through four 128-column TMEM buffers in issue order, and unit u
// belongs to issuer u & 1 and to warpgroup u & 1: two independent pipelines,
// each with one buffer being read and one being filled. Both issuers elect a thread
// of a uniform warp (ptx.cuh, elect_one): from one lane on per-thread registers the
// contractions set the pace at 740 cycles a unit (bf16; e4m3 470), now the epilogue
// does at 800 for 128 query rows, 500 for 32 (e4m3 item above: 121 -> 109 us). Eight epilogue warps keep
// the exponential unit as busy as sixteen do (4.8 cycles per 2^x and SM quarter
// against 4.0 at best) and leave 168 registers a thread for straight-line blocks
// of 64 columns: a branch per 32 columns (the reference check, the column count)
// kept a warp from overlapping one block's sums with the next one's exponents and
// cost 40% (P1 work per tile of two warps of an SM quarter: 1900 cycles, 1230 is
// the exponential unit's share).
// For e4m3 on long requests (choose_score_kernel has the line) an instance with four
// warpgroups, blocks of 32 columns and 96 registers: its contractions take half as
// long, and more warps hide the epilogue's latency (105.6 -> 98.7 us).
// Every wait is bounded (clock budget); on expiry the kernel sets the error
// word, drains its own copies and MMAs, frees TMEM and returns.

#include <math.h>

#include "internal.h"
#include "pipe.cuh"
#include "ptx.cuh"

namespace lvs {

namespace {

constexpr int kStatSlots = 4;  // stats of heads s-3..s may be live across the cluster
template <int N>
struct Blocks {
    static constexpr int value = N;
};
constexpr float kTileLimit = 4096.f;  // a tile that adds more to a pass-1 sum moves its reference

// Shared-memory plan. The ring gets whatever is left of the 227 KB after the
// Q double buffer and the bookkeeping; every variant needs more than half of
// the SM's shared memory, so a single CTA (and a single 512-column TMEM
// allocation) lives on an SM at a time.
template <int ROW_BYTES, int MROWS, int kEpiWG>
struct SmemLayout {
    static constexpr int KB = ROW_BYTES / 128;             // 128-byte swizzle blocks along d
    static constexpr int TILE_BYTES = kTileRows * ROW_BYTES;
    static constexpr int Q_BYTES = MROWS * ROW_BYTES;
    // Q(s) lives from pass 1 of head s to pass 2 of head s; a third buffer lets
    // Q(s+2) load while pass 2 of head s is still reading Q(s).
    static constexpr int QBUF = MROWS == 64 ? 3 : 2;
    static constexpr int FIXED = QBUF * Q_BYTES + kMaxTilesPerCta * kTileRows * 4 + kStatSlots * kMaxText * 8 +
                                 2 * kMaxText * 4 + 2 * (kEpiWG - 1) * kMaxText * 8 + 512 + 64 +
                                 1024;
    static constexpr int STAGES_FIT = (227 * 1024 - FIXED) / TILE_BYTES;
    // even: a stage then always belongs to the same issuer (unit u uses stage
    // u % kStages), which makes its waits on the stage's phases sound
    static constexpr int kStages = STAGES_FIT > 10 ? 10 : STAGES_FIT & ~1;
    static constexpr int OFF_K = 0;
    static constexpr int OFF_Q = OFF_K + kStages * TILE_BYTES;
    static constexpr int OFF_ACC = OFF_Q + QBUF * Q_BYTES;
    static constexpr int OFF_STATS = OFF_ACC + kMaxTilesPerCta * kTileRows * 4;
    static constexpr int OFF_B2 = OFF_STATS + kStatSlots * kMaxText * 8;
    static constexpr int OFF_XS = OFF_B2 + 2 * kMaxText * 4;  // [head & 1][kEpiWG - 1][128] float2: other warpgroups' row stats
    static constexpr int OFF_BAR = OFF_XS + 2 * (kEpiWG - 1) * kMaxText * 8;
    // k_full[S], k_empty[S], q_full[QBUF], q_empty[QBUF], u_full[4], u_empty[4],
    // stats[4], drain, stall, item_full[2], item_empty[2]
    static constexpr int NBAR = 2 * kStages + 2 * QBUF + 2 * 4 + kStatSlots + 2 + 4;
    static constexpr int OFF_ITEMS = OFF_BAR + NBAR * 8;  // [3][5] int: the items in work, the epilogue's
    static constexpr int OFF_MISC = OFF_ITEMS + 3 * 5 * 4;
    static constexpr int BYTES = OFF_MISC + 16;
    static constexpr int ALLOC = BYTES + 1024;  // slack for 1024-byte alignment
};

// An item as claimed, and what a CTA of its cluster serves of it.
struct TcItem {
    int hg, n0, N, t0, T;
};
struct TcWork {
    int hg, n0, N, t0, T;
    int R, n2;                     // query rows of a head block, rounded up to 16
    int tile_begin, tile_end, mt;
    // pass 1 runs with M = 64 for a request of at most 64 query rows, also in the
    // 128-row instance: its rows then lie in 16 lanes of each of the four lane
    // quadrants, so all SM sub-partitions work on them
    bool m64;
};

template <int kEpiWG>
constexpr int kThreadsOf = 96 + 128 * kEpiWG;

template <int ROW_BYTES, bool FP8, int MROWS, int kEpiWG>
__global__ void __launch_bounds__(kThreadsOf<kEpiWG>, 1)
    score_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                    const __grid_constant__ ScoreLaunch p)
{
    using L = SmemLayout<ROW_BYTES, MROWS, kEpiWG>;
    constexpr int kEpiThreads = 128 * kEpiWG, kThreads = kThreadsOf<kEpiWG>;
    constexpr int KSTEPS = ROW_BYTES / 32;                 // one MMA consumes 32 bytes of d
    constexpr int ELEMS_PER_KB = FP8 ? 128 : 64;           // elements in 128 bytes
    constexpr uint32_t FMT = FP8 ? 0u : 1u;
    constexpr int kStages = L::kStages;
    constexpr int QBUF = L::QBUF;
    static_assert(kStages >= 4 && kStages % 2 == 0, "ring depth");
    static_assert(L::ALLOC > 116 * 1024, "one CTA per SM");
    static_assert(L::ALLOC <= 227 * 1024, "shared memory per CTA");

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (base - raw);

    const int warp = uniform((int)(threadIdx.x >> 5)), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const uint32_t csize = cluster_nctarank();
    // With the full-key-set terms (p.extra, written by the kernel launched just
    // before this one) only the threads that read them wait for that kernel,
    // right before the read: this kernel's other inputs come from kernels that
    // had completed before that one passed its own wait, so the visual-key work
    // overlaps it. Every CTA still waits before it exits, so this grid never
    // completes ahead of that one.
    if (!p.extra) griddep_wait();
    griddep_launch_dependents();
    const bool multi = p.groups > 1;
    const int hp = p.hp;  // query heads of a head block
    const int G = p.hq / p.hkv;
    const int hpg = p.heads_per_group;
    const float cl = p.c_log2;
    // An item is a (request, head group); without a cluster a CTA works through
    // several, claimed in order of size (p.claims), and its roles run on from one
    // to the next: the copies and contractions of an item's first tiles lie under
    // the end of the one before.
    const bool shared = csize == 1 && (int)gridDim.x < p.items;  // items beyond each CTA's first
    auto make_work = [&](const TcItem& i) -> TcWork {
        TcWork w;
        w.hg = i.hg;
        w.n0 = i.n0;
        w.N = i.N;
        w.t0 = i.t0;
        w.T = i.T;
        w.R = i.T * hp;
        const int n_tiles = (i.N + kTileRows - 1) / kTileRows;
        const int tpc = (n_tiles + (int)csize - 1) / (int)csize;
        w.tile_begin = min(n_tiles, (int)rank * tpc);
        w.tile_end = min(n_tiles, w.tile_begin + tpc);
        w.mt = w.tile_end - w.tile_begin;
        w.n2 = (w.R + 15) & ~15;
        w.m64 = MROWS == 64 || w.R <= 64;
        return w;
    };
    // N = 0 for an item without work; shape errors are caught on the host, this
    // only keeps the kernel within its buffers
    auto get_item = [&](int item) -> TcItem {
        const int req_i = item / p.groups;
        const int b = p.order_n > 0 ? (int)p.order[req_i] : req_i;
        // the request's offsets: by value for small batches (no global load)
        const bool byv = p.nv > 0;
        TcItem i;
        i.hg = item - req_i * p.groups;
        i.n0 = byv ? p.so_v[b] : p.seq_off[b];
        i.N = (byv ? p.so_v[b + 1] : p.seq_off[b + 1]) - i.n0;
        const int tq = byv ? p.to_v[b] : p.text_off[b];
        const int t1 = byv ? p.to_v[b + 1] : p.text_off[b + 1];
        i.t0 = p.query_last && t1 > tq ? t1 - 1 : tq;  // last-token queries: one row
        i.T = t1 - i.t0;
        if (i.N > 0 && (i.T <= 0 || i.T * hp > MROWS || (i.N + kTileRows - 1) / kTileRows > kMaxTilesPerCta * (int)csize)) {
            atomicOr(p.err, kErrShape);
            i.N = 0;
        }
        return i;
    };
    TcWork mine{};  // the one item of a cluster
    if (csize > 1) {
        mine = make_work(get_item((int)(blockIdx.x / csize)));
        if (mine.N <= 0) {  // uniform for the whole cluster
            if (p.extra) griddep_wait();
            return;
        }
    }
    // Pass 2 of a head follows pass 1 of the next head (lag 1), so the
    // statistics exchange of the cluster overlaps a contraction; a CTA without
    // peers needs no exchange and runs both passes of a head in turn (lag 0),
    // which halves the K tiles that must stay in L2 for the re-read.
    const int lag = csize > 1 ? 1 : 0;

    const uint32_t bar0 = base + L::OFF_BAR;
    auto BAR = [&](int i) -> uint32_t { return bar0 + 8u * (uint32_t)i; };
    // U_FULL / U_EMPTY: a ring of four 128-column TMEM buffers shared by the
    // contractions of both passes, in issue order (unit u uses buffer u % 4)
    const int K_FULL = 0, K_EMPTY = kStages, Q_FULL = 2 * kStages, Q_EMPTY = Q_FULL + QBUF, U_FULL = Q_EMPTY + QBUF,
              U_EMPTY = U_FULL + 4, STATS = U_EMPTY + 4,
              DRAIN = STATS + kStatSlots, STALL = DRAIN + 1, IT_FULL = STALL + 1, IT_EMPTY = IT_FULL + 2;
    volatile int* items_s = reinterpret_cast<volatile int*>(smem + L::OFF_ITEMS);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::OFF_MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::OFF_MISC + 4);
    float* acc_s = reinterpret_cast<float*>(smem + L::OFF_ACC);
    float2* stats_s = reinterpret_cast<float2*>(smem + L::OFF_STATS);
    float* b2_s = reinterpret_cast<float*>(smem + L::OFF_B2);
    float2* xs_s = reinterpret_cast<float2*>(smem + L::OFF_XS);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(BAR(K_FULL + s), 1);
            mbar_init(BAR(K_EMPTY + s), 1);
        }
        for (int i = 0; i < QBUF; ++i) {
            mbar_init(BAR(Q_FULL + i), 1);
            mbar_init(BAR(Q_EMPTY + i), 2);  // one commit per issuer
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(BAR(U_FULL + i), 1);
            mbar_init(BAR(U_EMPTY + i), 4);  // one arrival per warp of the consuming warpgroup
        }
        for (int i = 0; i < kStatSlots; ++i) mbar_init(BAR(STATS + i), csize);
        mbar_init(BAR(DRAIN), 2);
        mbar_init(BAR(STALL), 1);  // nothing ever arrives (the debug stall below)
        for (int i = 0; i < 2; ++i) {
            mbar_init(BAR(IT_FULL + i), 1);
            mbar_init(BAR(IT_EMPTY + i), 3);  // the issuers and the epilogue
        }
        *abort_flag = 0;
        fence_mbar_init_cluster();
    }
    // Q rows past the copied box (MROWS not a multiple of hp) enter pass 2 as
    // columns whose terms are 2^-inf: they must be numbers
    for (int x = threadIdx.x; x < QBUF * L::KB * (MROWS - hp * p.box_rows) * 8; x += kThreads) {
        const int rows = MROWS - hp * p.box_rows, blk = x / (rows * 8), o = x - blk * (rows * 8);
        *reinterpret_cast<uint4*>(smem + L::OFF_Q + blk * MROWS * 128 + hp * p.box_rows * 128 + o * 16) =
            make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async_shared();
    }
    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&tm_q);
        tma_prefetch_desc(&tm_k);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // Cluster barrier, split: every thread arrives now (its CTA's barriers
    // exist) and waits only before its first remote arrival (the epilogue) or
    // before the final barrier (producer, MMA warp), so the first copies and
    // contractions do not wait for the slowest CTA of the cluster. The arrival
    // needs no release: the barriers' set-up is released by fence.mbarrier_init
    // above, and the statistics peers read are released by their own arrivals.
    cluster_arrive_relaxed();
    const uint32_t tmem = uniform(*tmem_slot);
    const Ctl ctl{abort_flag, p.err, p.wait_budget};

    // the k-th item of this CTA, for one thread of each role that follows the
    // producer; N = 0 when there is none, or after an abort
    auto take_item = [&](int k) -> TcItem {
        TcItem i{0, 0, 0, 0, 0};
        if (poll_phase(BAR(IT_FULL + (k & 1)), (uint32_t)(k >> 1) & 1u, ctl)) {
            const volatile int* q = items_s + (k & 1) * 5;
            i = TcItem{q[0], q[1], q[2], q[3], q[4]};
            mbar_arrive(BAR(IT_EMPTY + (k & 1)));
        }
        return i;
    };

    // Pipeline step s of an item (0..hpg): pass 1 of head s (s < hpg), then pass 2 of
    // head s - lag. hc counts the heads of the items before.
    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t ks = 0, kph = 0;
            int k_issued[kStages];
            int q_issued[QBUF];
            for (int s = 0; s < QBUF; ++s) q_issued[s] = 0;
            for (int s = 0; s < kStages; ++s) k_issued[s] = 0;
            // Debug stall (p.stall, a test of the failure path): wait on a barrier
            // that nothing completes before issuing any copy, so this wait runs out
            // of budget and every other wait of the launch runs out or sees the
            // abort flag, with no copy or contraction in flight.
            bool ok = !p.stall || poll_phase(BAR(STALL), 0, ctl);
            int item = (int)blockIdx.x, hc = 0;
            for (int k = 0; ok; ++k, hc += hpg) {
                TcWork w;
                if (csize > 1) {
                    if (k > 0 || mine.mt == 0) break;
                    w = mine;
                } else {
                    TcItem i{0, 0, 0, 0, 0};
                    if (k > 0) item = shared ? (int)gridDim.x + atomicAdd(p.claims, 1) : p.items;
                    while (item < p.items && (i = get_item(item)).N <= 0)
                        item = shared ? (int)gridDim.x + atomicAdd(p.claims, 1) : p.items;
                    if (!poll_phase(BAR(IT_EMPTY + (k & 1)), ((uint32_t)(k >> 1) & 1u) ^ 1u, ctl)) break;
                    volatile int* q = items_s + (k & 1) * 5;
                    q[0] = i.hg;
                    q[1] = i.n0;
                    q[2] = i.N;
                    q[3] = i.t0;
                    q[4] = i.T;
                    mbar_arrive(BAR(IT_FULL + (k & 1)));
                    if (i.N <= 0) break;  // the end, for every role
                    w = make_work(i);
                }
                auto load_tiles = [&](int g) {
                    for (int t = w.tile_begin; t < w.tile_end && ok; ++t) {
                        if (!poll_phase(BAR(K_EMPTY + ks), kph ^ 1, ctl)) { ok = false; break; }
                        mbar_arrive_expect_tx(BAR(K_FULL + ks), L::TILE_BYTES);
                        const uint32_t kdst = base + L::OFF_K + ks * L::TILE_BYTES;
#pragma unroll
                        for (int kb = 0; kb < L::KB; ++kb)
                            tma_load_3d(kdst + kb * kTileRows * 128, &tm_k, BAR(K_FULL + ks), kb * ELEMS_PER_KB, g,
                                        w.n0 + t * kTileRows);
                        ++k_issued[ks];
                        if (++ks == kStages) { ks = 0; kph ^= 1; }
                    }
                };
                for (int s = 0; s < hpg + lag && ok; ++s) {
                    if (s < hpg) {
                        const int h = (w.hg * hpg + s) * hp;
                        const int qb = (hc + s) % QBUF;
                        if (!poll_phase(BAR(Q_EMPTY + qb), ((uint32_t)((hc + s) / QBUF) & 1u) ^ 1u, ctl)) { ok = false; break; }
                        mbar_arrive_expect_tx(BAR(Q_FULL + qb), (uint32_t)(L::KB * 128 * hp * p.box_rows));
                        const uint32_t qdst = base + L::OFF_Q + qb * L::Q_BYTES;
#pragma unroll
                        for (int kb = 0; kb < L::KB; ++kb)
                            tma_load_3d(qdst + kb * MROWS * 128, &tm_q, BAR(Q_FULL + qb), kb * ELEMS_PER_KB, h, w.t0);
                        ++q_issued[qb];
                        load_tiles(h / G);
                    }
                    if (s >= lag && ok) load_tiles((w.hg * hpg + s - lag) * hp / G);
                }
            }
            // drain: the last load of every slot lands before the CTA leaves
            // (these waits ignore the abort flag)
            volatile int no_abort = 0;
            const Ctl drain_ctl{&no_abort, p.err, kWaitBudgetCycles};
            for (int s = 0; s < kStages; ++s)
                if (k_issued[s] > 0) poll_phase(BAR(K_FULL + s), (uint32_t)(k_issued[s] - 1) & 1u, drain_ctl);
            for (int s = 0; s < QBUF; ++s)
                if (q_issued[s] > 0) poll_phase(BAR(Q_FULL + s), (uint32_t)(q_issued[s] - 1) & 1u, drain_ctl);
        }
        __syncwarp();
        cluster_wait();
    } else if (warp <= 2) {
        // ------------------------------------------------------------ MMA issuers
        // Warps 1 and 2; issuer `who` takes the units u with (u & 1) == who, their
        // stages and TMEM buffers (both counts are even). The whole warp runs the
        // loop and an elected thread issues (elect_one). The operand descriptors
        // are made once per head (Q) and unit (K); each K step adds a constant to
        // the start-address field (shared-memory offsets stay below 256 KB, so the
        // 14-bit field never carries).
        const uint32_t who = (uint32_t)(warp - 1);
        const uint32_t idesc_r64 = idesc_make(64, 128, FMT), idesc_r128 = idesc_make(128, 128, FMT);
        uint32_t ks = 0, kph = 0, ui = 0;
        bool ok = true;
        int hc = 0;
        for (int k = 0; ok; ++k, hc += hpg) {
            if (csize > 1 && k > 0) break;
            TcItem item{mine.hg, mine.n0, mine.N, mine.t0, mine.T};
            if (csize == 1) {
                if (lane == 0) item = take_item(k);
                __syncwarp();
            }
            item = TcItem{uniform(item.hg), uniform(item.n0), uniform(item.N), uniform(item.t0), uniform(item.T)};
            const TcWork w = make_work(item);
            if (w.N <= 0 || w.mt == 0) break;
            const uint32_t idesc1 = w.m64 ? idesc_r64 : idesc_r128;
            const uint32_t idesc2 = idesc_make(128, (uint32_t)w.n2, FMT);
            for (int s = 0; s < hpg + lag && ok; ++s) {
                for (int pass = 0; pass < 2 && ok; ++pass) {
                    if (pass == 0 && s >= hpg) continue;
                    if (pass == 1 && s < lag) continue;
                    const int hs = hc + (pass == 0 ? s : s - lag);  // head of these units
                    const int qb = hs % QBUF;
                    if (pass == 0) {
                        if (!poll_phase_warp(BAR(Q_FULL + qb), (uint32_t)(hs / QBUF) & 1u, ctl)) { ok = false; break; }
                        tc_fence_after();
                    }
                    const uint64_t qdesc = sdesc_k_sw128(base + L::OFF_Q + qb * L::Q_BYTES);
                    for (int t = w.tile_begin; t < w.tile_end; ++t, ++ui) {
                        const uint32_t st_ks = ks, st_ph = kph;
                        if (++ks == kStages) { ks = 0; kph ^= 1; }
                        if ((ui & 1u) != who) continue;
                        const uint32_t ub = ui & 3, uph = (ui >> 2) & 1;
                        if (!poll_phase_warp(BAR(K_FULL + st_ks), st_ph, ctl) ||
                            !poll_phase_warp(BAR(U_EMPTY + ub), uph ^ 1, ctl)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint64_t kdesc = sdesc_k_sw128(base + L::OFF_K + st_ks * L::TILE_BYTES);
                        const uint32_t d = tmem + ub * 128u;
                        const uint64_t adesc = pass == 0 ? qdesc : kdesc, bdesc = pass == 0 ? kdesc : qdesc;
                        constexpr uint64_t kQ16 = MROWS * 128 / 16, kK16 = kTileRows * 128 / 16;
                        const uint64_t ablk = pass == 0 ? kQ16 : kK16, bblk = pass == 0 ? kK16 : kQ16;
                        const uint32_t idesc = pass == 0 ? idesc1 : idesc2;
                        if (elect_one()) {
#pragma unroll
                            for (int st = 0; st < KSTEPS; ++st) {
                                const uint64_t ad = adesc + (uint64_t)(st >> 2) * ablk + (uint64_t)(st & 3) * 2;
                                const uint64_t bd = bdesc + (uint64_t)(st >> 2) * bblk + (uint64_t)(st & 3) * 2;
                                if (FP8) mma_f8(d, ad, bd, idesc, st > 0);
                                else mma_f16(d, ad, bd, idesc, st > 0);
                            }
                            mma_commit(BAR(U_FULL + ub));
                            mma_commit(BAR(K_EMPTY + st_ks));
                        }
                        __syncwarp();
                    }
                    // Q(hs) is free once both issuers' contractions of its pass 2 are done
                    if (pass == 1 && ok) {
                        if (elect_one()) mma_commit(BAR(Q_EMPTY + qb));
                        __syncwarp();
                    }
                }
            }
        }
        // drain: every MMA issued by this warp's thread has completed
        if (elect_one()) mma_commit(BAR(DRAIN));
        __syncwarp();
        volatile int no_abort = 0;
        const Ctl drain_ctl{&no_abort, p.err, kWaitBudgetCycles};
        poll_phase_warp(BAR(DRAIN), 0, drain_ctl);
        cluster_wait();
    } else {
        // ------------------------------------------------------------ epilogue
        cluster_wait();  // the peers' barriers and buffers exist before any statistics go out
        // Two warpgroups; warpgroup wg takes the units u with (u & 1) == wg. A
        // unit's buffer was last used by unit u - 4 of the same warpgroup. Control
        // flow is identical within a warpgroup (named barriers); after an abort
        // every wait returns at once and the steps run out.
        const int quad = warp & 3;
        const int wg = (warp - 3) >> 2;                       // 0 .. kEpiWG - 1
        const int et = threadIdx.x - 96;                      // 0 .. kEpiThreads - 1
        const int wt = et & 127;
        const int vrow = quad * 32 + lane;                    // pass 2: TMEM lane = visual token in tile
        const uint32_t tcol = tmem + ((uint32_t)(quad * 32) << 16);
        const float2 cl2 = make_float2(cl, cl);
        // this warp has read buffer ub: hand it back
        auto release = [&](uint32_t ub) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(BAR(U_EMPTY + ub));
        };
        uint32_t ui = 0;  // contraction units in issue order (both passes)
        int hc = 0;
        // One thread takes the next item for all of them, so that every warp agrees on
        // it also when a wait gives up. It writes between two barriers of the
        // warpgroups that all readers of the item before have passed.
        volatile int* cur = items_s + 2 * 5;
        auto next_item = [&](int k) {
            if (csize == 1 && et == 0) {
                const TcItem i = take_item(k);
                cur[0] = i.hg;
                cur[1] = i.n0;
                cur[2] = i.N;
                cur[3] = i.t0;
                cur[4] = i.T;
            }
            named_bar_sync(1, kEpiThreads);
        };
        next_item(0);
        for (int k = 0;; hc += hpg) {
        const TcWork w = csize > 1 ? mine : make_work(TcItem{cur[0], cur[1], cur[2], cur[3], cur[4]});
        if (w.N <= 0) break;
        const int n0 = w.n0, N = w.N, t0 = w.t0, T = w.T, R = w.R, n2 = w.n2, mt = w.mt, hg = w.hg;
        const int tile_begin = w.tile_begin, tile_end = w.tile_end;
        const bool m64 = w.m64;
        // The units of an item come in pairs, so with four warpgroups its first may
        // belong to warpgroup 2: roles and the order of the merge below follow the
        // item's first unit, and its scores do not depend on the items before it.
        const int lead = kEpiWG == 4 ? (int)(ui & 3u) : 0;
        const int rwg = (wg - lead) & (kEpiWG - 1);
        // pass 1 row of this thread: M = 128 -> lane; M = 64 -> lanes 16q..16q+15, two
        // column halves
        const int prow = !m64 ? quad * 32 + lane : quad * 16 + (lane & 15);
        const bool p1_live = !m64 ? (quad * 32 < R) : (quad * 16 < R);
        for (int tl = wg; tl < mt; tl += kEpiWG) acc_s[tl * kTileRows + vrow] = 0.f;
        for (int s = 0; s < hpg + lag; ++s) {
            if (s < hpg) {
                // ---- pass 1 of head s: row sums over this warpgroup's tiles
                float ref = -INFINITY, nrc = 0.f;           // reference logit and -(ref * c), a whole number
                float2 s01 = make_float2(0.f, 0.f), s23 = make_float2(0.f, 0.f);
                // One tile: a row's columns (128; 64 with M = 64, the other 64 with the
                // thread 16 lanes on), in blocks of 64; `ld` reads 32 columns from c.
                auto tile = [&](auto ld, auto blocks, uint32_t ub, int valid, bool first, bool full) {
                    constexpr int NB = decltype(blocks)::value;
                    // columns past the request's end: 2^-inf adds nothing
                    auto ld_masked = [&](int c, float (&v)[32]) {
                        ld(c, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] = c + e < valid ? v[e] : -INFINITY;
                    };
                    auto sum_masked = [&]() {
#pragma unroll 1
                        for (int c = 0; c < NB * 64; c += 32) {
                            float v[32];
                            ld_masked(c, v);
                            row_sum_exp<32>(v, cl2, make_float2(nrc, nrc), s01, s23);
                        }
                    };
                    if (first) {
                        float v[32];
                        ld_masked(0, v);
                        ref = row_max<32>(v);
                        nrc = ref == -INFINITY ? 0.f : -rintf(ref * cl);
                    }
                    const float2 o01 = s01, o23 = s23;
                    const float before = (s01.x + s01.y) + (s23.x + s23.y);
                    if (full) {
#pragma unroll
                        for (int k = 0; k < (kEpiWG == 4 ? 2 * NB : 0); ++k) {
                            float v[32];
                            ld(k * 32, v);
                            tmem_wait_ld();
                            row_sum_exp<32>(v, cl2, make_float2(nrc, nrc), s01, s23);
                        }
#pragma unroll
                        for (int k = 0; k < (kEpiWG == 4 ? 0 : NB); ++k) {
                            float va[32], vb[32];
                            ld(k * 64, va);
                            ld(k * 64 + 32, vb);
                            tmem_wait_ld();
                            row_sum_exp<32>(va, cl2, make_float2(nrc, nrc), s01, s23);
                            row_sum_exp<32>(vb, cl2, make_float2(nrc, nrc), s01, s23);
                        }
                    } else {
                        sum_masked();
                    }
                    // a logit far above the reference (or not a number), or no reference
                    // yet: take the tile's maximum into the reference and redo the tile
                    const float added = (s01.x + s01.y) + (s23.x + s23.y) - before;
                    if (__any_sync(0xffffffffu, !(added < kTileLimit) || ref == -INFINITY)) {
                        float m = ref;
#pragma unroll 1
                        for (int c = 0; c < NB * 64; c += 32) {
                            float v[32];
                            ld_masked(c, v);
                            m = fmaxf(m, row_max<32>(v));
                        }
                        const float nr = m == -INFINITY ? 0.f : -rintf(m * cl);
                        const float f = ref == -INFINITY ? 0.f : ex2(nr - nrc);
                        ref = m;
                        nrc = nr;
                        s01 = make_float2(o01.x * f, o01.y * f);
                        s23 = make_float2(o23.x * f, o23.y * f);
                        sum_masked();
                    }
                    release(ub);
                };
                bool started = false;  // a tile of this row has been summed (warp-uniform)
                for (int t = tile_begin; t < tile_end; ++t, ++ui) {
                    if ((int)(ui % kEpiWG) != wg) continue;
                    const uint32_t ub = ui & 3;
                    poll_phase(BAR(U_FULL + ub), (ui >> 2) & 1, ctl);
                    tc_fence_after();
                    if (!p1_live) {
                        release(ub);
                        continue;
                    }
                    const uint32_t ta = tcol + ub * 128u;
                    const int left = N - t * kTileRows;  // columns of the request in this tile
                    const bool first = !started, full = left >= kTileRows;
                    started = true;
                    if (MROWS == 128 && !m64)
                        tile([&](int c, float* v) { tmem_ld32(ta + (uint32_t)c, v); }, Blocks<2>{}, ub, left, first, full);
                    else
                        tile([&](int c, float* v) { tmem_ld16x2_32<64>(ta + (uint32_t)c, v); }, Blocks<1>{}, ub,
                             left - (lane >> 4) * 64, first, full);
                }
                // the reference in units of log2, as the sums used it
                float m = ref == -INFINITY ? ref : -nrc, l = (s01.x + s01.y) + (s23.x + s23.y);
                if (m64) {
                    // merge the two column parts of each row (threads t and t ^ 16)
                    const float mo = __shfl_xor_sync(0xffffffffu, m, 16);
                    const float lo = __shfl_xor_sync(0xffffffffu, l, 16);
                    merge_row(m, l, mo, lo);
                }
                // ---- merge the warpgroups, publish (m, l) of head s to the cluster
                const bool writer = !m64 || lane < 16;
                // (double-buffered by head: the other warpgroups may publish head s + 1
                // while the first one is still reading head s)
                float2* xs = xs_s + ((hc + s) & 1) * (kEpiWG - 1) * kMaxText;
                if (rwg > 0 && writer) xs[(rwg - 1) * kMaxText + prow] = make_float2(m, l);
                named_bar_sync(1, kEpiThreads);
                if (rwg == 0) {
                    if (writer) {
#pragma unroll
                        for (int o_wg = 1; o_wg < kEpiWG; ++o_wg) {  // fixed order: deterministic
                            const float2 o = xs[(o_wg - 1) * kMaxText + prow];
                            merge_row(m, l, o.x, o.y);
                        }
                        stats_s[((hc + s) % kStatSlots) * kMaxText + prow] = make_float2(m, l);
                    }
                    named_bar_sync(2, 128);
                    // one release arrival per CTA of the cluster, each from its own
                    // thread: a release at cluster scope covers the rows the other
                    // threads wrote before the named barrier, and the arrivals'
                    // fences (each waits for this SM's memory traffic to settle)
                    // overlap instead of running one after another
                    if (csize > 1 && wt < (int)csize)
                        mbar_arrive_remote(mapa_shared(BAR(STATS + s % kStatSlots), (uint32_t)wt));
                }
            }
            if (s >= lag) {
                // ---- merge the cluster's statistics of head s - lag
                const int hs = s - lag;
                const int slot = (hc + hs) % kStatSlots;
                float* b2 = b2_s + ((hc + hs) & 1) * kMaxText;
                if (rwg == 0) {
                    // (a CTA that is its own cluster reads its own rows, ordered by the named barrier above)
                    if (csize > 1) poll_phase<true>(BAR(STATS + slot), (uint32_t)(hs / kStatSlots) & 1u, ctl);
                    if (wt < R) {
                        const uint32_t row = (uint32_t)(slot * kMaxText + wt);
                        const float2 st = csize > 1 ? merge_cluster_row(base + L::OFF_STATS + row * 8u, csize) : stats_s[row];
                        // For e4m3 the logarithm's error is a good part of a score's: mean
                        // relative error over 8 draws of 13 requests of up to 3248 tokens
                        // 1.34e-7 with __log2f and 1.19e-7 with log2f (0.97e-7 in the resident
                        // kernel that had this call), of 32 of up to 3456 1.04e-7 and 0.81e-7,
                        // at the same time. For bf16 and with other keys' terms it offsets
                        // another one (12 requests, 32 / 8 heads: 1.5e-7, 2.3e-7 with log2f).
                        float bm = st.x + (FP8 && !p.extra ? log2f(st.y) : __log2f(st.y));
                        if (p.extra) {
                            griddep_wait();
                            bm = log2_add(bm, p.extra[(int64_t)(t0 + wt / hp) * p.hq + (hg * hpg + hs) * hp + wt % hp]);
                        }
                        b2[wt] = -bm;  // stored negated: the fma addend of pass 2
                    } else {
                        b2[wt] = -INFINITY;
                    }
                }
                named_bar_sync(1, kEpiThreads);
                // ---- pass 2 of head hs: per-visual-token sums of probabilities
                for (int t = tile_begin; t < tile_end; ++t, ++ui) {
                    if ((int)(ui % kEpiWG) != wg) continue;
                    const uint32_t ub = ui & 3;
                    poll_phase(BAR(U_FULL + ub), (ui >> 2) & 1, ctl);
                    tc_fence_after();
                    float2 a01 = make_float2(0.f, 0.f), a23 = make_float2(0.f, 0.f);
                    const uint32_t ta = tcol + ub * 128u;
#pragma unroll
                    for (int c0 = 0; c0 < (kEpiWG == 4 ? MROWS : 0); c0 += 32) {
                        if (n2 >= c0 + 32) {
                            float v[32];
                            tmem_ld32(ta + (uint32_t)c0, v);
                            tmem_wait_ld();
                            if (n2 == c0 + 32) release(ub);
                            col_sum_exp16(v, cl2, b2 + c0, a01, a23);
                            col_sum_exp16(v + 16, cl2, b2 + c0 + 16, a01, a23);
                        } else if (n2 > c0) {  // the last 16
                            float v[16];
                            tmem_ld16(ta + (uint32_t)c0, v);
                            tmem_wait_ld();
                            release(ub);
                            col_sum_exp16(v, cl2, b2 + c0, a01, a23);
                        }
                    }
#pragma unroll
                    for (int c0 = 0; c0 < (kEpiWG == 4 ? 0 : MROWS); c0 += 64) {
                        if (n2 >= c0 + 64) {  // a straight-line block of 64 columns
                            float va[32], vb[32];
                            tmem_ld32(ta + (uint32_t)c0, va);
                            tmem_ld32(ta + (uint32_t)(c0 + 32), vb);
                            tmem_wait_ld();
                            if (n2 == c0 + 64) release(ub);
                            col_sum_exp16(va, cl2, b2 + c0, a01, a23);
                            col_sum_exp16(va + 16, cl2, b2 + c0 + 16, a01, a23);
                            col_sum_exp16(vb, cl2, b2 + c0 + 32, a01, a23);
                            col_sum_exp16(vb + 16, cl2, b2 + c0 + 48, a01, a23);
                        } else if (n2 > c0) {  // the last 16, 32 or 48
                            float va[32], vb[16];
                            tmem_ld32(ta + (uint32_t)c0, va);
                            tmem_ld16(ta + (uint32_t)(c0 + 32), vb);
                            tmem_wait_ld();
                            release(ub);
                            col_sum_exp16(va, cl2, b2 + c0, a01, a23);
                            if (n2 > c0 + 16) col_sum_exp16(va + 16, cl2, b2 + c0 + 16, a01, a23);
                            if (n2 > c0 + 32) col_sum_exp16(vb, cl2, b2 + c0 + 32, a01, a23);
                        }
                    }
                    acc_s[(t - tile_begin) * kTileRows + vrow] += (a01.x + a01.y) + (a23.x + a23.y);
                }
            }
        }
        next_item(++k);  // (with its barrier every tile's sums are in acc_s)
        // ---- results
        const float denom = (float)p.hq * (float)T;
        for (int tl = wg; tl < mt; tl += kEpiWG) {
            const int j = (tile_begin + tl) * kTileRows + vrow;
            if (j < N) {
                const float a = acc_s[tl * kTileRows + vrow];
                if (!multi) p.out[n0 + j] = a / denom;
                else p.partials[(int64_t)hg * p.total_vis + n0 + j] = a;
            }
        }
        if (csize > 1) break;
        }
        tc_fence_before();
    }

    // ---------------------------------------------------------------- teardown
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
    if (p.extra) griddep_wait();  // returns at once for threads that already waited
    cluster_sync_all();  // peers are done reading this CTA's statistics
    // the last CTA to leave clears the claims for the next launch
    if (shared && threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(p.claims + 1, 1) == (int)gridDim.x - 1) p.claims[0] = p.claims[1] = 0;
    }
}

// scores = sum over the head groups' partial rows, in group order, / (Hq * T):
// grid (256-token chunks of the longest request, requests)
constexpr int kFoldThreads = 256;

__global__ void __launch_bounds__(kFoldThreads) fold_kernel(const __grid_constant__ FoldArgs a)
{
    griddep_wait();
    griddep_launch_dependents();
    for (int b = blockIdx.y; b < a.batch; b += gridDim.y) {
        const int n0 = a.nv > 0 ? a.so_v[b] : a.seq_off[b];
        const int N = (a.nv > 0 ? a.so_v[b + 1] : a.seq_off[b + 1]) - n0;
        const int j = blockIdx.x * kFoldThreads + threadIdx.x;
        if (j >= N) continue;
        const int T = a.query_last ? 1 : (a.nv > 0 ? a.to_v[b + 1] - a.to_v[b] : a.text_off[b + 1] - a.text_off[b]);
        const float* src = a.partials + n0 + j;
        float sum = 0.f;
        for (int g = 0; g < a.groups; g += 16) {
            float v[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] = g + q < a.groups ? __ldcg(src + (int64_t)(g + q) * a.total_vis) : 0.f;
#pragma unroll
            for (int q = 0; q < 16; ++q)
                if (g + q < a.groups) sum += v[q];
        }
        a.out[n0 + j] = sum / ((float)a.hq * (float)T);
    }
}

template <int ROW_BYTES, bool FP8, int MROWS, int kEpiWG = 2>
cudaError_t tc_prepare(int cluster)
{
    auto kern = score_tc_kernel<ROW_BYTES, FP8, MROWS, kEpiWG>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         SmemLayout<ROW_BYTES, MROWS, kEpiWG>::ALLOC);
    if (e == cudaSuccess && cluster > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// CTAs resident at once with clusters of `cluster` CTAs (occupancy query)
template <int ROW_BYTES, bool FP8, int MROWS, int kEpiWG = 2>
int tc_capacity(int cluster)
{
    if (tc_prepare<ROW_BYTES, FP8, MROWS, kEpiWG>(cluster) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster * 64, 1, 1);
    cfg.blockDim = dim3(kThreadsOf<kEpiWG>, 1, 1);
    cfg.dynamicSmemBytes = SmemLayout<ROW_BYTES, MROWS, kEpiWG>::ALLOC;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, score_tc_kernel<ROW_BYTES, FP8, MROWS, kEpiWG>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n * cluster;
}

template <int ROW_BYTES, bool FP8, int MROWS, int kEpiWG = 2>
cudaError_t launch_variant(const CUtensorMap& tm_q, const CUtensorMap& tm_k, const ScoreLaunch& p,
                           const ScorePlan& plan, int batch, cudaStream_t stream)
{
    auto kern = score_tc_kernel<ROW_BYTES, FP8, MROWS, kEpiWG>;
    const int smem = SmemLayout<ROW_BYTES, MROWS, kEpiWG>::ALLOC;
    cudaError_t e = tc_prepare<ROW_BYTES, FP8, MROWS, kEpiWG>(plan.cluster);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    // clusters: one per item; without, as many CTAs as run at once, which share the items
    // (or one per item, where the call has no claims)
    const int items = plan.groups * batch;
    const int ctas = plan.cluster > 1 || !p.claims || items < plan.ctas ? plan.cluster * items : plan.ctas;
    cfg.gridDim = dim3((unsigned)ctas, 1, 1);
    cfg.blockDim = dim3(kThreadsOf<kEpiWG>, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = plan.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = pdl_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, tm_q, tm_k, p);
}

}  // namespace

int tc_cluster_capacity(int row_bytes, bool fp8, int mrows, int cluster)
{
    if (fp8) return mrows == 64 ? tc_capacity<128, true, 64>(cluster) : tc_capacity<128, true, 128>(cluster);
    if (row_bytes == 256)
        return mrows == 64 ? tc_capacity<256, false, 64>(cluster) : tc_capacity<256, false, 128>(cluster);
    return mrows == 64 ? tc_capacity<128, false, 64>(cluster) : tc_capacity<128, false, 128>(cluster);
}

bool score_shape_supported(int head_dim, bool fp8)
{
    if (fp8) return head_dim == 128;
    return head_dim == 64 || head_dim == 128;
}

// Launch shape of the re-read kernel with the lowest modelled time.
ScorePlan plan_score(const BatchTiles& bt, int hq, int hkv, int row_bytes, const int* cap_by_cluster,
                     const KernelCosts& costs, double window_one, double* cost_out)
{
    ScorePlan best{1, 1, 1};
    double best_cost = 1e300;
    const int max_tiles = bt.n > 0 ? bt.desc[0] : 0;
    if (max_tiles <= 0) {
        if (cost_out) *cost_out = 0.0;
        return best;
    }
    const int G = hq / hkv;
    const double tile_bytes = (double)kTileRows * row_bytes;
    double rows = 0.0;
    for (int i = 0; i < bt.n; ++i) rows += (double)bt.desc[i] * kTileRows;
    for (int pass = 0; pass < 2 && best_cost >= 1e299; ++pass) {
        for (int c = 1; c <= kMaxCluster; ++c) {
            const int tpc = (max_tiles + c - 1) / c;
            if (tpc > kMaxTilesPerCta) continue;
            if (c > 1 && (c - 1) * tpc >= max_tiles) continue;  // an idle rank on the largest request
            const int cap = cap_by_cluster[c];
            if (cap < c) continue;
            for (int g = 1; g <= hq; ++g) {
                if (hq % g) continue;
                const long long ctas = (long long)bt.n * c * g;
                const int hpg = hq / g;
                // L2 window of the pass-2 re-read: while a CTA streams a slice (in a
                // cluster up to two: pass 1 of the next head, rest of the current one)
                // the tiles it re-reads must survive in L2. Groups that split a GQA
                // key head share its tiles. The bound is loose (160 MB against 126 MB
                // of L2): the re-read follows pass 1 within one head, and whole-request
                // CTAs measured faster than clusters of two up to there (full keys,
                // 16 requests of 4 to 21 tiles: 39.1 against 42.6 us).
                const long long active = ctas < cap ? ctas : cap;
                const int share = hpg >= G ? 1 : G / hpg;
                const double window = (c > 1 ? 2.0 : window_one) * tpc * tile_bytes * (double)active / share;
                if (pass == 0 && window > 160.0 * 1024 * 1024) continue;
                // beyond 110 MB some of the re-read comes from HBM: 32 requests of 27
                // tiles, 32 heads (134 MB) took 264 us where the tiles alone make 190
                const double miss = costs.fold_once && window > 110e6 ? 1.0 + (window - 110e6) / 110e6 : 1.0;
                auto item_cost = [&](int tiles) {
                    const int t = (tiles + c - 1) / c;
                    return tiles <= 0 ? costs.empty
                                      : (c > 1 ? costs.start : costs.next) + (g > 1 && !costs.fold_once ? costs.fold : 0.0) +
                                            hpg * (t * costs.tile * miss + (c > 1 ? costs.exchange : costs.exchange_one));
                };
                // a fold of its own also moves the partial rows once out and in
                const double cost = makespan(bt, g, cap / c, item_cost) + (c > 1 ? 0.0 : costs.start - costs.next) +
                                    (g > 1 && costs.fold_once ? costs.fold + g * rows * 8.0 / 4e6 : 0.0);
                if (cost < best_cost - 1e-9) {
                    best_cost = cost;
                    best = ScorePlan{c, tpc, g};
                    best.ctas = cap;
                }
            }
        }
    }
    if (cost_out) *cost_out = best_cost;
    return best;
}

cudaError_t launch_fold(const FoldArgs& a, int max_n, cudaStream_t stream)
{
    if (a.batch <= 0 || max_n <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((max_n + kFoldThreads - 1) / kFoldThreads), (unsigned)(a.batch < 65535 ? a.batch : 65535), 1);
    cfg.blockDim = dim3(kFoldThreads, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fold_kernel, a);
}

cudaError_t launch_score(const CUtensorMap& tm_q, const CUtensorMap& tm_k, const ScoreLaunch& p,
                         const ScorePlan& plan, int batch, int row_bytes, bool fp8, int mrows, cudaStream_t stream)
{
    ScoreLaunch q = p;
    q.groups = plan.groups;
    q.hp = plan.hp;
    q.box_rows = mrows / plan.hp;
    q.heads_per_group = p.hq / plan.hp / plan.groups;
    q.ctas_per_request = plan.cluster * plan.groups;
    q.items = plan.groups * batch;
    if (plan.cluster == 1 && plan.ctas < 1) return cudaErrorInvalidValue;
    if (fp8) {
        if (plan.wide)
            return mrows == 64 ? launch_variant<128, true, 64, 4>(tm_q, tm_k, q, plan, batch, stream)
                               : launch_variant<128, true, 128, 4>(tm_q, tm_k, q, plan, batch, stream);
        return mrows == 64 ? launch_variant<128, true, 64>(tm_q, tm_k, q, plan, batch, stream)
                           : launch_variant<128, true, 128>(tm_q, tm_k, q, plan, batch, stream);
    }
    if (row_bytes == 256) {
        return mrows == 64 ? launch_variant<256, false, 64>(tm_q, tm_k, q, plan, batch, stream)
                           : launch_variant<256, false, 128>(tm_q, tm_k, q, plan, batch, stream);
    }
    return mrows == 64 ? launch_variant<128, false, 64>(tm_q, tm_k, q, plan, batch, stream)
                       : launch_variant<128, false, 128>(tm_q, tm_k, q, plan, batch, stream);
}

}  // namespace lvs

// Attention core on compacted heads (Eq. 2 per head, with the heads of the coupled-matrix reformulation of Sec. 3.1
// restricted to their kept indices): Ctx_h = softmax(scale * Q_h K_h^T) V_h for heads whose Q/K width and V width
// differ from head to head, forward and backward.  sm_100a: TMA tile loads -> shared memory -> tcgen05.mma with the
// score tiles and the output tile in TMEM; the softmax runs in registers, one thread per query row.
//
// Layout: Q^c, K^c (T x n_qk) and V^c, Ctx (T x n_vo) hold head h in columns [off_h, off_h + w_h) with w_h a multiple of
// 16 (the compaction step pads every head's block with zero columns: a zero column of Q^c / K^c adds nothing to
// Q K^T, and a zero column of V^c gives a zero column of Ctx) and off_h a multiple of 8, so that every tile load starts
// on a 16-byte boundary and every contraction is a whole number of 16-deep MMA steps.
//
// Two forward kernels, one CTA per SM.  Output heads up to 32 wide (with Q/K heads up to 64) take the kernel of independent key
// streams further down (attn_fwd_ms_kernel) unless there are many sequences of up to two tiles (the rule stands in
// ecospa_coupled_attn_fwd); all others take the kernel described here, 640 threads.
// A work item is one or two tiles of 128 query rows, one per stream (see FwdItems); a CTA walks a static list of items (for
// causal attention the long ones first).  Two neighbouring query tiles of a sequence and head share the K / V tiles.
//   warp 0       one lane issues the TMA loads of the streams' Q tiles and of the K / V tiles (rings of 4 or 2 stages); a tile
//                is one or two 64-column blocks of 128 rows x 128 bytes, 128-byte swizzle
//   warps 1, 2   one lane each issues the products of its stream: S = Q K^T (K-major operands from shared memory) and
//                O += P V (P read from TMEM, V as stored = MN-major), accumulating in TMEM
//   warps 4..11  scaling, four warps per stream: where a key block raises a row's maximum, the output row so far is multiplied by
//                2^(m_old - m_new) while the softmax warps exponentiate; at the end of an item times 1 / l and to memory
//   warps 12..19 softmax, four warps per stream; thread = query row = TMEM lane, all 128 key columns, so nothing is exchanged
//                between threads.  A first pass over the scores takes the row maximum, a second one p = 2^(s*c - m), which it
//                packs to bf16 and writes to TMEM for the second product.  Every probability is taken against the row's running
//                maximum, so the largest one of a row is exactly 1.
// Both passes are rolled loops of 64 columns: holding a block's 128 scores in registers, unrolled, was slower (163 -> 233 us at
// 4 x 2048 positions, 32 heads 32 wide: warps waited for instructions, 4.0 of 15 cycles per issue, now 1.0).  Columns that
// no row of a warp sees are skipped, keys past the end of the sequence also in the products.
// Before (two streams in one thread's registers, a token between them) / now, us: 475 / 301 (2 x 4096, 32 heads 96 wide),
// 69.7 / 53.2 (4 x 1000, 32 heads 48 wide on 8), 10.5 / 7.5 (2 x 160, 12 heads 48 wide), 63.3 / 26.8 (60 x 48, 32 heads 64
// wide), 41.7 / 18.3 (30 x 48, 32 heads 128 wide), 26.4 / 24.7 (8 x 512, 16 heads 64 wide, no mask).  One form is slower than before: one
// pair of tiles to a CTA, short, without a mask, heads of 33 to 64 (9.7 / 10.3 for 96 heads of 256, 12.2 / 12.6 for 72 of 384): the two
// streams start and end together.
// Every mbarrier wait is bounded; on expiry the CTA records a code (11 loads, 12 products, 13 softmax and scaling) in the device
// status word, lets copies land, frees TMEM and returns.

#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "gemm.cuh"
#include "tc.cuh"

namespace ecospa {

namespace {

using namespace tc;

constexpr int kTile = 128;                  // query rows and key rows per tile
constexpr int kBlockBytes = kTile * 128;    // one 64-column block of a 128-row tile
constexpr int kMaxHeads = 128;
constexpr int kFwdThreads = 640;              // four service warps; per stream four scaling and four softmax warps
constexpr int kBwdComputeWarps = 16;
constexpr int kBwdThreads = 64 + 4 * 128 + 64;   // producer warp, MMA warp, four sets of four compute warps, two more MMA warps
constexpr int kTmemCols = 512;

struct HeadLayout {
    int32_t qk_off[kMaxHeads], qk_w[kMaxHeads], vo_off[kMaxHeads], vo_w[kMaxHeads];   // per query head: Q^c and Ctx columns, widths
    int32_t k_off[kMaxHeads], v_off[kMaxHeads];   // per query head: first column of its K/V head in K^c and in V^c
    int32_t rep;                                   // query heads per K/V head (1: every head its own)
};

struct AttnFwdParams {
    alignas(64) CUtensorMap map_q, map_k, map_v;
    HeadLayout heads;
    int32_t batch, seq, n_heads, n_qt, causal, n_items;
    int32_t items;                          // FwdItems
    int32_t turns;                          // wide heads: the two streams exponentiate in turn
    float scale_log2e;                      // scale * log2(e): scores are exponentiated in base 2
    uint16_t* ctx;
    int64_t ld_ctx;
    float* lse;                             // [n_heads][T], natural logarithm
    int* status;
    unsigned long long wait_limit_ns;
};

// Work items are listed long ones first (causal attention) and dealt to the CTAs in rounds that run through the list
// alternately forwards and backwards: with a plain stride the first CTA gets the longest item of every round.  (32 query
// heads on 8 K/V heads, 4 x 1000 positions, dK and dV: 48 steps for the first CTA where the mean is 31; 87 -> 75 us.)
__device__ __forceinline__ int dealt_item(uint32_t round) {
    const int r = static_cast<int>(round), G = gridDim.x, c = blockIdx.x;
    return (r & 1) ? (r + 1) * G - 1 - c : r * G + c;
}

// A work item is one or two tiles of 128 query rows, one per stream.
enum FwdItems {
    ITEMS_SHARED = 0,   // two neighbouring query tiles of a (sequence, head); both streams read the same K / V tiles
    ITEMS_SOLO = 1,     // sequences of one tile: two (sequence, head) units, each with a K / V tile of its own
    ITEMS_SINGLE = 2,   // one query tile (few of them: each gets an SM to itself)
};
struct FwdItem {
    int h0, b0, qt0, n0, h1, b1, qt1, n1;   // of stream 0 and 1: head, sequence, query tile, key blocks (0: no such tile)
};
__device__ __forceinline__ FwdItem decode_item(int it, const AttnFwdParams& P) {
    FwdItem I;
    const int per = P.n_heads * P.batch;
    if (P.items == ITEMS_SOLO) {
        const int u0 = 2 * it, u1 = min(u0 + 1, per - 1);
        I.h0 = u0 / P.batch;
        I.b0 = u0 % P.batch;
        I.h1 = u1 / P.batch;
        I.b1 = u1 % P.batch;
        I.qt0 = I.qt1 = 0;
        I.n0 = 1;
        I.n1 = u0 + 1 < per ? 1 : 0;
        return I;
    }
    const int rem = it % per, a = it / per;
    I.h0 = I.h1 = rem / P.batch;
    I.b0 = I.b1 = rem % P.batch;
    if (P.items == ITEMS_SINGLE) {
        I.qt0 = I.qt1 = P.n_qt - 1 - a;                            // long (late) query tiles first
        I.n1 = 0;
    } else {                                                       // (an odd one out is the first, the shortest)
        const int qa = 2 * ((P.n_qt + 1) / 2 - 1 - a) - (P.n_qt & 1);
        I.qt0 = max(qa, 0);
        I.qt1 = qa + 1;
        I.n1 = qa < 0 ? 0 : (P.causal ? qa + 2 : P.n_qt);
    }
    I.n0 = P.causal ? I.qt0 + 1 : P.n_qt;
    return I;
}

template <int NB>   // 64-column blocks per tile: 1 (every head at most 64 wide) or 2
struct FwdCfg {
    static constexpr int kTileBytes = NB * kBlockBytes;
    static constexpr int QS = NB == 1 ? 2 : 1;                     // buffers of a stream's Q tile
    static constexpr int ST = NB == 1 ? 4 : 2;                     // stages of the K and of the V tiles
    static constexpr int kRowBytes = (2 * 2 + 2 * 2) * kTile * 4;  // [buffer][stream][row]: factor of the outputs, then 1 / sum
    static constexpr int kOutBytes = 8 * 32 * 64;                  // output rows on their way out: [scaling warp][row][32 columns]
    static constexpr int kSmem = (2 * QS + 2 * ST) * kTileBytes + kRowBytes + kOutBytes + 1024 + 512;
    static constexpr int kOCols = NB * 64;                          // columns of an output tile
    // TMEM columns of stream x: scores, output, probabilities (narrow heads: a region of their own, so that the scores of the
    // next key block are computed while these are made; wide heads: over the scores they were made from)
    static __device__ __forceinline__ uint32_t col_s(uint32_t x) { return 128u * x; }
    static __device__ __forceinline__ uint32_t col_o(uint32_t x) { return 256u + kOCols * x; }
    static __device__ __forceinline__ uint32_t col_p(uint32_t x) { return NB == 1 ? 384u + 64u * x : 128u * x; }
    static constexpr bool kEarly = NB == 1;                         // scores one block ahead of the probabilities
    static_assert(kSmem <= 232448, "shared memory of a block");
};

template <int NB, bool STAGED>   // STAGED: output rows leave through shared memory
__global__ void __launch_bounds__(kFwdThreads, 1) attn_fwd_kernel(const __grid_constant__ AttnFwdParams P) {
    using Cfg = FwdCfg<NB>;
    constexpr int kTileBytes = Cfg::kTileBytes, QS = Cfg::QS, ST = Cfg::ST;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (base - raw_addr);
    const uint32_t sQ = base, sK = sQ + 2 * QS * kTileBytes, sV = sK + ST * kTileBytes;   // Q: [stage][stream]
    float* row_factor = reinterpret_cast<float*>(smem + (2 * QS + 2 * ST) * kTileBytes);    // [buffer][stream][row]
    float* row_inv = row_factor + 4 * kTile;                                                // [buffer][stream][row]
    const uint32_t sOut = base + (2 * QS + 2 * ST) * kTileBytes + Cfg::kRowBytes;
    uint8_t* tail = smem + (2 * QS + 2 * ST) * kTileBytes + Cfg::kRowBytes + Cfg::kOutBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(tail);
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(tail + 52 * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 52 * 8 + 8);
    const uint32_t bar0 = smem_u32(bars);
    auto q_full = [&](uint32_t x, uint32_t s) { return bar0 + 8u * (2 * x + s); };
    auto q_empty = [&](uint32_t x, uint32_t s) { return bar0 + 8u * (4 + 2 * x + s); };
    auto k_full = [&](uint32_t s) { return bar0 + 8u * (8 + s); };
    auto k_empty = [&](uint32_t s) { return bar0 + 8u * (12 + s); };
    auto v_full = [&](uint32_t s) { return bar0 + 8u * (16 + s); };
    auto v_empty = [&](uint32_t s) { return bar0 + 8u * (20 + s); };
    // per stream: scores complete; scores in registers; product with the probabilities done.  In pairs, used alternately, where
    // a warp may arrive for one step before every other has looked at the step before: probabilities and rescaled output ready,
    // factors of the rows written, sums of the rows written.
    auto s_full = [&](uint32_t x) { return bar0 + 8u * (24 + x); };
    auto s_read = [&](uint32_t x) { return bar0 + 8u * (26 + x); };
    auto pv_done = [&](uint32_t x) { return bar0 + 8u * (28 + x); };
    auto p_full = [&](uint32_t x, uint32_t b) { return bar0 + 8u * (30 + 2 * x + b); };
    auto f_full = [&](uint32_t x, uint32_t b) { return bar0 + 8u * (34 + 2 * x + b); };
    auto l_full = [&](uint32_t x, uint32_t b) { return bar0 + 8u * (38 + 2 * x + b); };
    // whose turn it is to exponentiate, per scheduler: warp q of stream 0 and warp q of stream 1 share one
    auto turn_of = [&](uint32_t x, uint32_t q) { return bar0 + 8u * (42 + 4 * x + q); };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (uint32_t x = 0; x < 2; ++x) {
            for (uint32_t s = 0; s < 2; ++s) {
                mbar_init(q_full(x, s), 1);
                mbar_init(q_empty(x, s), 1);
                mbar_init(p_full(x, s), 8);       // (one arrival per softmax warp and per scaling warp of the stream)
                mbar_init(f_full(x, s), 4);
                mbar_init(l_full(x, s), 4);
            }
            mbar_init(s_full(x), 1);
            mbar_init(s_read(x), 4);
            mbar_init(pv_done(x), 1);
            for (uint32_t q = 0; q < 4; ++q) mbar_init(turn_of(x, q), 1);
        }
        for (uint32_t s = 0; s < 4; ++s) {
            mbar_init(k_full(s), 1);
            mbar_init(k_empty(s), 2);             // both streams
            mbar_init(v_full(s), 1);
            mbar_init(v_empty(s), 2);
        }
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tensormap(&P.map_q);
        prefetch_tensormap(&P.map_k);
        prefetch_tensormap(&P.map_v);
    }
    pdl_start();
    if (warp == 1) tmem_alloc(smem_u32(tmem_holder), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    pdl_wait();

    // K / V stage and phase of a tile (solo: tiles and stages are numbered per stream)
    const bool solo = P.items == ITEMS_SOLO;
    auto stage = [&](uint32_t tile, uint32_t x) -> uint32_t { return solo ? 2 * (tile % (ST / 2)) + x : tile % ST; };
    auto phase = [&](uint32_t tile) -> uint32_t { return (solo ? tile / (ST / 2) : tile / ST) & 1u; };

    if (warp == 0) {
        // ------------------------------------------------------------------ loads
        if (elect_one()) {
            uint32_t t = 0, round = 0;                              // K / V tiles (solo: of a stream) and items before this item
            bool ok = true;
            auto load_q = [&](uint32_t x, uint32_t n, int h, int row) -> bool {
                const uint32_t qs = n % QS;
                if (!mbar_wait(q_empty(x, qs), ((n / QS) & 1u) ^ 1u, abort_flag, 11, P.status, P.wait_limit_ns)) return false;
                const int nb = (P.heads.qk_w[h] + 63) >> 6;
                mbar_expect_tx(q_full(x, qs), nb * kBlockBytes);
                for (int blk = 0; blk < nb; ++blk)
                    tma_load_2d(sQ + (2 * qs + x) * kTileBytes + blk * kBlockBytes, &P.map_q, P.heads.qk_off[h] + 64 * blk, row, q_full(x, qs));
                return true;
            };
            uint32_t nq0 = 0, nq1 = 0;
            for (int it = dealt_item(0); ok && it < P.n_items; it = dealt_item(++round)) {
                const FwdItem I = decode_item(it, P);
                ok = load_q(0, nq0++, I.h0, I.b0 * P.seq + I.qt0 * kTile);
                if (ok && I.n1 > 0) ok = load_q(1, nq1++, I.h1, I.b1 * P.seq + I.qt1 * kTile);
                const int tiles = solo ? 1 + I.n1 : max(I.n0, I.n1);
                for (int j = 0; ok && j < tiles; ++j) {
                    const bool second = solo && j == 1;
                    const uint32_t tile = solo ? t : t + j, st = stage(tile, second), ph = phase(tile) ^ 1u;
                    const int h = second ? I.h1 : I.h0, y = (second ? I.b1 : I.b0) * P.seq + (solo ? 0 : j * kTile);
                    const int nbq = (P.heads.qk_w[h] + 63) >> 6, nbv = (P.heads.vo_w[h] + 63) >> 6;
                    if (!(ok = mbar_wait(k_empty(st), ph, abort_flag, 11, P.status, P.wait_limit_ns))) break;
                    mbar_expect_tx(k_full(st), nbq * kBlockBytes);
                    for (int blk = 0; blk < nbq; ++blk)
                        tma_load_2d(sK + st * kTileBytes + blk * kBlockBytes, &P.map_k, P.heads.k_off[h] + 64 * blk, y, k_full(st));
                    if (!(ok = mbar_wait(v_empty(st), ph, abort_flag, 11, P.status, P.wait_limit_ns))) break;
                    mbar_expect_tx(v_full(st), nbv * kBlockBytes);
                    for (int blk = 0; blk < nbv; ++blk)
                        tma_load_2d(sV + st * kTileBytes + blk * kBlockBytes, &P.map_v, P.heads.v_off[h] + 64 * blk, y, v_full(st));
                }
                t += solo ? 1 : tiles;
            }
        }
    } else if (warp < 3) {
        // ------------------------------------------------------------------ products of stream x
        // The stream goes through all the tiles of its CTA, also those that only the other one uses (it hands them back unused).
        const uint32_t x = warp - 1;
        if (!(P.items == ITEMS_SINGLE && x == 1) && elect_one()) {
            uint32_t nq = 0, ns = 0, np = 0;                        // items, score tiles and probability tiles of this stream so far
            bool ok = true;
            // the tile a step works on: tile number, widths of the head, key block, and how many of the item's key blocks are this stream's
            struct Slot {
                uint32_t tile;
                int wq, wv, j, n, n_max;
                bool valid;
            };
            uint32_t round = 0;
            auto item_start = [&](Slot& d) {
                const int it = dealt_item(round);
                d.valid = it < P.n_items;
                if (!d.valid) return;
                const FwdItem I = decode_item(it, P);
                d.wq = P.heads.qk_w[x ? I.h1 : I.h0];
                d.wv = P.heads.vo_w[x ? I.h1 : I.h0];
                d.j = 0;
                d.n = x ? I.n1 : I.n0;
                d.n_max = solo ? 1 : max(I.n0, I.n1);
                if (solo && d.n == 0) d.valid = false;               // (the odd unit out is the last item's)
            };
            auto release = [&](uint32_t bar) {                      // once the products issued so far are done
                tc_commit(bar);
                if (P.items != ITEMS_SHARED) tc_commit(bar);         // (in the other stream's place)
            };
            // S_x = Q_x K^T.  On narrow heads the scores of the step before must be in registers; on wide heads this comes after the
            // product that read the probabilities made from them.
            auto scores = [&](const Slot& d) -> bool {
                const uint32_t st = stage(d.tile, x);
                if (!mbar_wait(k_full(st), phase(d.tile), abort_flag, 12, P.status, P.wait_limit_ns)) return false;
                if (d.j >= d.n) {
                    mbar_arrive(k_empty(st));
                    return true;
                }
                const uint32_t qs = nq % QS;
                if (d.j == 0 && !mbar_wait(q_full(x, qs), (nq / QS) & 1u, abort_flag, 12, P.status, P.wait_limit_ns)) return false;
                const int steps = d.wq >> 4, cols = min(kTile, P.seq - d.j * kTile);     // keys of the tile, in whole steps of 16
                const uint32_t idesc = make_idesc(kTile, (cols + 15) & ~15, 0, 0);
                const uint64_t dq = make_smem_desc(sQ + (2 * qs + x) * kTileBytes, 16, 1024), dk = make_smem_desc(sK + st * kTileBytes, 16, 1024);
                // (the wait that decides when the products can go comes last, with all their operands at hand)
                if (Cfg::kEarly && ns > 0 && !mbar_wait(s_read(x), (ns - 1) & 1u, abort_flag, 12, P.status, P.wait_limit_ns)) return false;
                ++ns;
                tc_fence_after();
#pragma unroll
                for (int ks = 0; ks < 4 * NB; ++ks) {
                    const uint32_t o = ((ks >> 2) * kBlockBytes + (ks & 3) * 32) >> 4;
                    if (ks < steps) tc_mma_bf16(tmem_base + Cfg::col_s(x), dq + o, dk + o, idesc, ks != 0 ? 1u : 0u);
                }
                tc_commit(s_full(x));
                release(k_empty(st));
                if (d.j == d.n - 1) {
                    tc_commit(q_empty(x, qs));
                    ++nq;
                }
                return true;
            };
            // O_x (+)= P_x V over the keys of the tile
            auto outputs = [&](const Slot& d) -> bool {
                const uint32_t st = stage(d.tile, x);
                if (!mbar_wait(v_full(st), phase(d.tile), abort_flag, 12, P.status, P.wait_limit_ns)) return false;
                if (d.j >= d.n) {
                    mbar_arrive(v_empty(st));
                    return true;
                }
                const int steps = (min(kTile, P.seq - d.j * kTile) + 15) >> 4;
                const uint32_t idesc = make_idesc(kTile, d.wv, 0, 1);
                const uint64_t dv = make_smem_desc(sV + st * kTileBytes, kBlockBytes, 1024);
                if (!mbar_wait(p_full(x, np & 1u), (np >> 1) & 1u, abort_flag, 12, P.status, P.wait_limit_ns)) return false;
                ++np;
                tc_fence_after();
#pragma unroll
                for (int ks = 0; ks < kTile / 16; ++ks)
                    if (ks < steps) tc_mma_bf16_ts(tmem_base + Cfg::col_o(x), tmem_base + Cfg::col_p(x) + 8 * ks, dv + 128 * ks, idesc, (d.j | ks) != 0 ? 1u : 0u);
                tc_commit(pv_done(x));
                release(v_empty(st));
                return true;
            };
            Slot cur, nxt;
            cur.valid = false;
            nxt.tile = 0;
            item_start(nxt);
            while (ok && (cur.valid || nxt.valid)) {
                if (Cfg::kEarly && nxt.valid) ok = scores(nxt);
                if (ok && cur.valid) ok = outputs(cur);
                if (ok && !Cfg::kEarly && nxt.valid) ok = scores(nxt);
                cur = nxt;
                if (nxt.valid) {
                    ++nxt.tile;
                    if (++nxt.j == nxt.n_max) {
                        ++round;
                        item_start(nxt);
                    }
                }
            }
        }
    } else if (warp >= 4 && warp < 12) {
        // ------------------------------------------------------------------ scaling of the outputs of stream x
        const uint32_t x = static_cast<uint32_t>(warp - 4) >> 2;
        const int row = (warp & 3) * 32 + lane;
        const uint32_t tO = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) + Cfg::col_o(x);
        uint32_t ns = 0, nf = 0, nl = 0, round = 0;                  // steps, factors, items of this stream so far
        bool ok = true;
        for (int it = dealt_item(0); ok && it < P.n_items; it = dealt_item(++round)) {
            const FwdItem I = decode_item(it, P);
            const int n_own = x ? I.n1 : I.n0, h = x ? I.h1 : I.h0, wv = P.heads.vo_w[h];
            if (n_own == 0) continue;
            for (int j = 0; j < n_own; ++j, ++ns) {
                if (j > 0) {
                    if (!(ok = mbar_wait(f_full(x, nf & 1u), (nf >> 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
                    const float a = row_factor[((nf & 1u) * 2 + x) * kTile + row];
                    ++nf;
                    if (__any_sync(0xffffffffu, a != 1.f)) {         // some row of the warp has a new maximum
                        if (!(ok = mbar_wait(pv_done(x), (ns - 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
                        tc_fence_after();
                        const f32x2 a2 = pack2(a, a);
#pragma unroll 1
                        for (int c = 0; c < wv; c += 16) {
                            uint32_t r[16];
                            tc_ld16(tO + c, r);
                            tc_wait_ld(r);
#pragma unroll
                            for (int i = 0; i < 16; i += 2) {
                                float u, v;
                                unpack2(mul2(pack2(r[i], r[i + 1]), a2), u, v);
                                r[i] = __float_as_uint(u);
                                r[i + 1] = __float_as_uint(v);
                            }
                            tc_st(tO + c, r);
                        }
                        tc_wait_st();
                        tc_fence_before();
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(p_full(x, ns & 1u));
            }
            if (!ok) break;
            // the item's output rows: times 1 / sum, to memory
            if (!(ok = mbar_wait(l_full(x, nl & 1u), (nl >> 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
            if (!(ok = mbar_wait(pv_done(x), (ns - 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
            tc_fence_after();
            const float inv = row_inv[((nl & 1u) * 2 + x) * kTile + row];
            ++nl;
            const int q_warp = (x ? I.qt1 : I.qt0) * kTile + (warp & 3) * 32;
            uint16_t* dst = P.ctx + (static_cast<int64_t>(x ? I.b1 : I.b0) * P.seq + q_warp) * P.ld_ctx + P.heads.vo_off[h];
            if constexpr (STAGED) {
                // 32 columns at a time, eight rows to a store instruction
                const uint32_t buf = sOut + (warp - 4) * 2048;                // [row][4 chunks of 8 columns], chunk c of row r in place c ^ (r / 2 % 4)
                const int r_in = lane >> 2, chunk = lane & 3;                 // on the way out: eight rows to an instruction, four lanes to a row
#pragma unroll 1
                for (int c = 0; c < wv; c += 32) {
                    uint32_t r[16], q[16];                                     // (columns past the head's width are not stored)
                    tc_ld16(tO + c, r);
                    tc_ld16(tO + c + 16, q);
                    tc_wait_ld(r);
                    tc_wait_ld(q);
                    __syncwarp();                                              // the columns before these have left
                    auto put = [&](const uint32_t (&v)[16], int at, int k) {
                        st_shared_v4(buf + lane * 64 + 16 * (k ^ ((lane >> 1) & 3)), pack_bf16(__uint_as_float(v[at]) * inv, __uint_as_float(v[at + 1]) * inv),
                                     pack_bf16(__uint_as_float(v[at + 2]) * inv, __uint_as_float(v[at + 3]) * inv),
                                     pack_bf16(__uint_as_float(v[at + 4]) * inv, __uint_as_float(v[at + 5]) * inv),
                                     pack_bf16(__uint_as_float(v[at + 6]) * inv, __uint_as_float(v[at + 7]) * inv));
                    };
                    put(r, 0, 0);
                    put(r, 8, 1);
                    put(q, 0, 2);
                    put(q, 8, 3);
                    __syncwarp();
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int rr = 8 * u + r_in;
                        if (q_warp + rr < P.seq && c + 8 * chunk < wv)
                            *reinterpret_cast<uint4*>(dst + rr * P.ld_ctx + c + 8 * chunk) = ld_shared_v4(buf + rr * 64 + 16 * (chunk ^ ((rr >> 1) & 3)));
                    }
                }
            } else {
                const int q_pos = q_warp + lane;
#pragma unroll 1
                for (int c = 0; c < wv; c += 16) {
                    uint32_t r[16];
                    tc_ld16(tO + c, r);
                    tc_wait_ld(r);
                    if (q_pos < P.seq) {
                        uint4 v0, v1;
                        v0.x = pack_bf16(__uint_as_float(r[0]) * inv, __uint_as_float(r[1]) * inv);
                        v0.y = pack_bf16(__uint_as_float(r[2]) * inv, __uint_as_float(r[3]) * inv);
                        v0.z = pack_bf16(__uint_as_float(r[4]) * inv, __uint_as_float(r[5]) * inv);
                        v0.w = pack_bf16(__uint_as_float(r[6]) * inv, __uint_as_float(r[7]) * inv);
                        v1.x = pack_bf16(__uint_as_float(r[8]) * inv, __uint_as_float(r[9]) * inv);
                        v1.y = pack_bf16(__uint_as_float(r[10]) * inv, __uint_as_float(r[11]) * inv);
                        v1.z = pack_bf16(__uint_as_float(r[12]) * inv, __uint_as_float(r[13]) * inv);
                        v1.w = pack_bf16(__uint_as_float(r[14]) * inv, __uint_as_float(r[15]) * inv);
                        *reinterpret_cast<uint4*>(dst + lane * P.ld_ctx + c) = v0;
                        *reinterpret_cast<uint4*>(dst + lane * P.ld_ctx + c + 8) = v1;
                    }
                }
            }
            tc_fence_before();
        }
    } else if (warp >= 12) {
        // ------------------------------------------------------------------ softmax of stream x
        const uint32_t x = static_cast<uint32_t>(warp - 12) >> 2;
        const int row = (warp & 3) * 32 + lane;
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const uint32_t tS = t_lane + Cfg::col_s(x), tP = t_lane + Cfg::col_p(x);
        // Wide heads: the streams exponentiate in turn, warp by warp.  Both at once they take as long for it, and then wait for their
        // products at the same time too; the scores of narrow heads come a block ahead, and the turns cost more than they give.  (2 x
        // 4096, 32 heads 96 wide 358 -> 335 us, 16 x 512, 80 wide, no mask 99 -> 88; 8 x 1024, 48 wide: 100 -> 120.)
        const bool turns = NB == 2 && P.turns;
        uint32_t turn = 0;
        auto take_turn = [&]() -> bool {
            return !turns || mbar_wait(turn_of(x, warp & 3), x == 0 ? (turn & 1u) ^ 1u : turn & 1u, abort_flag, 13, P.status, P.wait_limit_ns);
        };
        auto pass_turn = [&]() {
            if (!turns) return;
            ++turn;
            __syncwarp();
            if (lane == 0) mbar_arrive(turn_of(x ^ 1u, warp & 3));
        };
        uint32_t ns = 0, nf = 0, nl = 0, round = 0;                         // steps, factors, items of this stream so far
        bool ok = true;
        for (int it = dealt_item(0); ok && it < P.n_items; it = dealt_item(++round)) {
            const FwdItem I = decode_item(it, P);
            const int n_own = x ? I.n1 : I.n0;
            if (n_own == 0 && !turns) continue;
            const int q_base = (x ? I.qt1 : I.qt0) * kTile, q_pos = q_base + row;   // position of this row in its sequence
            const int limit = P.causal ? min(P.seq, q_pos + 1) : P.seq;     // keys [0, limit) are visible to the row,
            const int w_limit = P.causal ? min(P.seq, q_base + ((warp & 3) + 1) * 32) : P.seq;   // and these to some row of the warp
            const int w_first = P.causal ? min(P.seq, q_base + (warp & 3) * 32 + 1) : P.seq;     // every row of the warp sees these
            float m = -INFINITY, l = 0.f;
            for (int j = 0; j < n_own; ++j, ++ns) {
                const int kv_base = j * kTile;
                // columns with a visible key, and those that the product reads (zeros beyond the first)
                const int n_vis = min(kTile, w_limit - kv_base), n_pv = min(kTile, P.seq - kv_base);
                if (!(ok = mbar_wait(s_full(x), ns & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
                tc_fence_after();
                // row maximum, 64 columns at a time; keys past the limit count as -inf (and are left so for the second pass)
                float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
                for (int c = 0; c < n_vis; c += 64) {
                    uint32_t a[32], b[32];
                    tc_ld32(tS + c, a);
                    tc_ld32(tS + c + 32, b);
                    tc_wait_ld(a);
                    tc_wait_ld(b);
                    if (kv_base + c + 64 > w_first) {
                        const int vis = limit - kv_base - c;
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            if (i >= vis) a[i] = 0xff800000u;
                            if (i + 32 >= vis) b[i] = 0xff800000u;
                        }
                        tc_st32(tS + c, a);
                        tc_st32(tS + c + 32, b);
                        tc_wait_st();
                    }
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        mx4[(i >> 1) & 1] = max3(mx4[(i >> 1) & 1], __uint_as_float(a[i]), __uint_as_float(a[i + 1]));
                        mx4[2 + ((i >> 1) & 1)] = max3(mx4[2 + ((i >> 1) & 1)], __uint_as_float(b[i]), __uint_as_float(b[i + 1]));
                    }
                }
                const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
                const float m_new = fmaxf(m, mx * P.scale_log2e), alpha = ex2(m - m_new);
                if (j > 0) {                                                // the output row is rescaled while this thread exponentiates
                    row_factor[((nf & 1u) * 2 + x) * kTile + row] = alpha;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(f_full(x, nf & 1u));
                    ++nf;
                }
                ok = take_turn();
                if (!ok) break;
                // p = 2^(s * c - m_new), packed to bf16, and the row sum
                float sum[4] = {0.f, 0.f, 0.f, 0.f};
                auto exponentiate = [&](uint32_t (&a)[32]) {               // 32 scores -> 16 packed pairs, in place
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        const float p0 = ex2(fmaf(__uint_as_float(a[i]), P.scale_log2e, -m_new)), p1 = ex2(fmaf(__uint_as_float(a[i + 1]), P.scale_log2e, -m_new));
                        sum[i & 2] += p0;
                        sum[(i & 2) + 1] += p1;
                        a[i >> 1] = pack_bf16(p0, p1);
                    }
                };
                int c = 0;
#pragma unroll 1
                for (; c < n_vis; c += 64) {
                    uint32_t a[32], b[32];
                    tc_ld32(tS + c, a);
                    tc_ld32(tS + c + 32, b);
                    tc_wait_ld(a);
                    tc_wait_ld(b);
                    if (Cfg::kEarly && c + 64 >= n_vis) {                   // the last of the scores are in registers
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(s_read(x));
                    }
                    exponentiate(a);
                    if (Cfg::kEarly && c == 0 && ns > 0) {                  // the last probabilities have been read (wide heads: the scores came after that product)
                        ok = mbar_wait(pv_done(x), (ns - 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns);
                        tc_fence_after();
                    }
                    tc_st16(tP + (c >> 1), a);
                    exponentiate(b);
                    tc_st16(tP + (c >> 1) + 16, b);
                }
                if (c < n_pv) {                                             // (at most 64 columns that only later rows see)
                    uint32_t z[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) z[i] = 0u;
                    tc_st32(tP + (c >> 1), z);
                }
                if (!ok) break;
                pass_turn();
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(p_full(x, ns & 1u));
                l = fmaf(l, alpha, (sum[0] + sum[1]) + (sum[2] + sum[3]));
                m = m_new;
            }
            for (int j = n_own; turns && ok && j < max(I.n0, I.n1); ++j) {   // (a stream without a tile left lets the other one go on)
                ok = take_turn();
                pass_turn();
            }
            if (!ok) break;
            if (n_own == 0) continue;
            row_inv[((nl & 1u) * 2 + x) * kTile + row] = 1.f / l;
            __syncwarp();
            if (lane == 0) mbar_arrive(l_full(x, nl & 1u));
            ++nl;
            if (q_pos < P.seq)
                P.lse[(static_cast<int64_t>(x ? I.h1 : I.h0) * P.batch + (x ? I.b1 : I.b0)) * P.seq + q_pos] = m * 0.6931471805599453f + logf(l);
        }
    }

    // ---------------------------------------------------------------------- teardown
    __syncwarp();
    if (*abort_flag) {
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);   // copies still in flight land before the memory is released
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// ------------------------------------------------------------------------------------------------
// forward, output heads up to 32 wide, not many short sequences: NS independent streams per CTA
// (EXACT: a slice's maximum is taken before its exponentials and the reference is the stream's running maximum; see the rule in
// ecospa_coupled_attn_fwd.  Otherwise one pass over the scores, against a reference that moves when a score exceeds it by 2^32.)
// ------------------------------------------------------------------------------------------------
// A work item is (sequence b, head h, one tile of 128 query rows).  A K / V tile holds NS slices of 64 keys; stream x
// (four warps, thread = query row) owns slice x of every tile and keeps a softmax of its own over its keys: reference
// exponent m_x, sum l_x, and the output O_x = sum_j P_x(j) V_x(j) accumulating in TMEM.  At the end of the item the NS
// partial results of a row are merged (M = max m_x, weights 2^(m_x - M)).  The streams never wait for one another inside
// an item, so while one waits for its products the others keep the exponential unit busy.
// One pass per score slice: p = 2^(s*c - m) with the reference m the stream already has; m moves only when a score
// exceeds it by more than 32 (2^32 headroom in fp32 / bf16, whose relative precision does not depend on the scale; the row's
// largest probability is rounded like the others, not exactly 1), in which case the row's l, O and the probabilities already
// written for the slice are rescaled first, so no exponent can overflow.  The first slice of an item starts from m = -1e30 and takes that path once.
// A stream has two score buffers: S_x of slice G + 1 is computed while the stream exponentiates slice G, so a stream goes
// from one slice to the next without waiting for the tensor pipe.  The probabilities of a slice overwrite the first half
// of the score buffer they were made from (chunk c of 32 scores becomes 16 packed columns at 16 c, inside columns
// that are already in registers).  TMEM columns of stream x: score buffers at 128 x and 128 x + 64, output 128 NS + OC x.
template <int NS, int OC>
struct MsCfg {
    // per stream: one warp that loads the stream's K / V slices and issues its products, and four softmax warps
    static constexpr int kThreads = 32 * NS + 128 * NS;
    static constexpr int kSlice = 64;
    static constexpr int kKeys = NS * kSlice;                 // keys per K / V tile
    static constexpr int kSliceBytes = kSlice * 128;          // one slice: 64 rows x 128 bytes
    static constexpr int kStages = 3;                         // K and V slices per stream: slice s uses stage s % 3
    static constexpr int kRingBytes = NS * 2 * kStages * kSliceBytes;
    static constexpr int kMergeBytes = 2 * NS * kTile * 4;    // m and l of every stream and row
    static constexpr int kSmem = 2 * kBlockBytes + kRingBytes + kMergeBytes + 1024 + 512;
    static __device__ __forceinline__ uint32_t col_s(uint32_t x, uint32_t buf) { return 128u * x + 64u * buf; }
    static __device__ __forceinline__ uint32_t col_o(uint32_t x) { return 128u * NS + OC * x; }
    static_assert(128 * NS + OC * NS <= kTmemCols, "TMEM columns");
};

struct MsItem {
    int b, h, qt, lim;          // lim: last key position any row of the tile sees
};
__device__ __forceinline__ MsItem ms_decode(int it, int n_qt, int n_heads, int batch, int seq, int causal) {
    MsItem I;
    const int per = n_heads * batch;
    I.qt = n_qt - 1 - it / per;             // long (late) query tiles first
    const int rem = it % per;
    I.h = rem / batch;
    I.b = rem % batch;
    I.lim = causal ? min(I.qt * kTile + kTile - 1, seq - 1) : seq - 1;
    return I;
}
// K / V tiles in which slice x has a visible key
__device__ __forceinline__ int ms_steps(int lim, int x, int keys_per_tile) {
    const int first = 64 * x;
    return lim >= first ? (lim - first) / keys_per_tile + 1 : 0;
}

struct RowState {
    float m, l, rs;
};
// The rare path of a slice: a score exceeds the row's reference exponent by more than 32.  Moves the reference to that
// score and rescales what was computed with the old one: the sums, the output row in TMEM (o_groups 16-column groups; 0
// while the stream has no output yet) and the probability chunks of this slice written so far.  Called by whole warps.
__device__ __forceinline__ RowState rescale_row(RowState s, float cm, uint32_t tO, int o_groups, uint32_t tP, int chunks_done) {
    const bool need = cm - s.m > 32.f;
    const float m_new = need ? cm : s.m;
    const float f = need ? ex2(s.m - m_new) : 1.f;
    tc_wait_st();                            // the chunks written so far are read back below
    for (int g = 0; g < o_groups; ++g) {
        uint32_t r[16];
        tc_ld16(tO + 16 * g, r);
        tc_wait_ld(r);
#pragma unroll
        for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * f);
        tc_st(tO + 16 * g, r);
    }
    for (int c = 0; c < chunks_done; ++c) {
        uint32_t r[16];
        tc_ld16(tP + 16 * c, r);
        tc_wait_ld(r);
#pragma unroll
        for (int i = 0; i < 16; ++i) r[i] = pack_bf16(bf16_lo(r[i]) * f, bf16_hi(r[i]) * f);
        tc_st(tP + 16 * c, r);
    }
    tc_wait_st();
    RowState o;
    o.m = m_new;
    o.l = s.l * f;
    o.rs = s.rs * f;
    return o;
}

template <int NS, int OC, bool EXACT>
__global__ void __launch_bounds__(MsCfg<NS, OC>::kThreads, 1) attn_fwd_ms_kernel(const __grid_constant__ AttnFwdParams P) {
    using Cfg = MsCfg<NS, OC>;
    constexpr int kSliceB = Cfg::kSliceBytes, kKeys = Cfg::kKeys, ST = Cfg::kStages;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (base - raw_addr);
    const uint32_t sQ = base, sK = sQ + 2 * kBlockBytes, sV = sK + NS * ST * kSliceB;   // K / V: [stream][stage] slices
    float* merge = reinterpret_cast<float*>(smem + 2 * kBlockBytes + Cfg::kRingBytes);   // [m | l][stream][row]
    uint8_t* tail = smem + 2 * kBlockBytes + Cfg::kRingBytes + Cfg::kMergeBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(tail);
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(tail + 60 * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 60 * 8 + 8);
    const uint32_t bar0 = smem_u32(bars);
    auto q_full = [&](uint32_t s) { return bar0 + 8u * s; };
    auto q_empty = [&](uint32_t s) { return bar0 + 8u * (2 + s); };     // one arrival per stream and item
    // Per stream and score buffer (slice G uses buffer G & 1): probabilities written; the product that read them done.
    // Two barriers each, because a stream runs ahead of its issuer by one slice: with one barrier the phases of slices
    // G and G + 1 could both complete before the waiter has looked at the first.
    auto p_full = [&](uint32_t x, uint32_t buf) { return bar0 + 8u * (4 + 2 * x + buf); };
    auto pv_done = [&](uint32_t x, uint32_t buf) { return bar0 + 8u * (42 + 2 * x + buf); };
    auto s_full = [&](uint32_t x, uint32_t buf) { return bar0 + 8u * (12 + 2 * x + buf); };   // scores in buffer buf of stream x
    auto kv_full = [&](uint32_t x, uint32_t b) { return bar0 + 8u * (20 + 2 * x + b); };      // the loads event G needs (b = G & 1) landed
    auto k2_full = [&](uint32_t x) { return bar0 + 8u * (48 + x); };                          // the third K slice of stream x landed
    const uint32_t merge_a = bar0 + 8u * 40, merge_b = bar0 + 8u * 41;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (uint32_t x = 0; x < NS; ++x) mbar_init(k2_full(x), 1);
        for (uint32_t s = 0; s < 2; ++s) {
            mbar_init(q_full(s), 1);
            mbar_init(q_empty(s), NS);
            for (uint32_t x = 0; x < NS; ++x) {
                mbar_init(kv_full(x, s), 1);
                mbar_init(s_full(x, s), 1);
                mbar_init(p_full(x, s), 128);
                mbar_init(pv_done(x, s), 1);
            }
        }
        mbar_init(merge_a, 128 * NS);
        mbar_init(merge_b, 128 * NS);
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tensormap(&P.map_q);
        prefetch_tensormap(&P.map_k);
        prefetch_tensormap(&P.map_v);
    }
    pdl_start();
    if (warp == 0) tmem_alloc(smem_u32(tmem_holder), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    pdl_wait();

    if (warp < NS) {
        // ------------------------------------------------------------------ loader and MMA issuer of stream x
        // The stream's slices form one sequence G = 0, 1, ... across the CTA's items (items in which the stream has no
        // visible key are skipped).  Event G: the probabilities of slice G are written -> O_x += P_x V_x (slice G), then
        // S_x of slice G + 2 into the score buffer that slice G occupied, then the loads of the K slice G + 3 and of the V
        // slice G + 1.  Their stages (slice s uses stage s % 3) are free: S(G) was read by the softmax, and P V(G - 2) was
        // issued before S(G), whose completion signal covers it.  Both loads report to the barrier event G + 1 waits on.
        // This thread shares its scheduler with the stream's softmax warps, so the loop is kept short: slices are
        // described by a few registers produced once (next()) and handed from stage to stage.
        if (elect_one()) {
            const uint32_t x = warp;
            const uint32_t tS = tmem_base + Cfg::col_s(x, 0), tO = tmem_base + Cfg::col_o(x);
            const uint32_t idesc_s = make_idesc(kTile, 64, 0, 0);
            const uint32_t sKx = sK + x * ST * kSliceB, sVx = sV + x * ST * kSliceB;
            const uint64_t dq0 = make_smem_desc(sQ, 16, 1024), dk0 = make_smem_desc(sKx, 16, 1024),
                           dv0 = make_smem_desc(sVx, kBlockBytes, 1024);
            // meta bits: 0 valid (clear: the end mark), 1 first slice of its item, 2 last, 3 Q buffer, 4 phase of that buffer,
            // 5-7 contraction steps of the scores, 8-11 output width / 16
            struct SD {
                int row;            // first key row of the slice in the K / V tensors
                int qrow;           // first row of the item's query tile
                uint32_t qcol;      // first column of the head in Q^c
                uint32_t kcol, vcol;   // first column of the head's K/V head in K^c and in V^c
                uint32_t meta;
            };
            // generator of the stream's slice sequence
            int g_it = 0, g_J = 0, g_n = 0, g_row = 0, g_qrow = 0;
            uint32_t g_kcol = 0, g_vcol = 0, g_qcol = 0, g_meta = 0, g_qi = ~0u, g_skip = 0;
            auto next = [&]() {
                SD d;
                if (g_J >= g_n) {
                    for (;;) {
                        g_it = dealt_item(++g_qi);
                        if (g_it >= P.n_items) {   // end mark
                            d.row = 0;
                            d.kcol = d.vcol = 0;
                            d.qcol = 0;
                            d.meta = 0;
                            --g_qi;                 // stay at the end: later calls give the mark again
                            g_J = g_n = 0;
                            d.qrow = 0;
                            return d;
                        }
                        const MsItem I = ms_decode(g_it, P.n_qt, P.n_heads, P.batch, P.seq, P.causal);
                        g_n = ms_steps(I.lim, x, kKeys);
                        if (g_n == 0) {
                            ++g_skip;
                            continue;
                        }
                        g_J = 0;
                        g_row = I.b * P.seq + 64 * static_cast<int>(x);
                        g_qrow = I.b * P.seq + I.qt * kTile;
                        g_kcol = static_cast<uint32_t>(P.heads.k_off[I.h]);
                        g_vcol = static_cast<uint32_t>(P.heads.v_off[I.h]);
                        g_qcol = static_cast<uint32_t>(P.heads.qk_off[I.h]);
                        g_meta = 1u | ((g_qi & 1u) << 3) | (((g_qi >> 1) & 1u) << 4) | (static_cast<uint32_t>(P.heads.qk_w[I.h] >> 4) << 5) |
                                 (static_cast<uint32_t>(P.heads.vo_w[I.h] >> 4) << 8);
                        break;
                    }
                }
                d.row = g_row + g_J * kKeys;
                d.qrow = g_qrow;
                d.qcol = g_qcol;
                d.kcol = g_kcol;
                d.vcol = g_vcol;
                d.meta = g_meta | (g_J == 0 ? 2u : 0u) | (g_J == g_n - 1 ? 4u : 0u);
                ++g_J;
                return d;
            };
            bool ok = true;
            // K slice of d into stage st (stream 0: with the Q tile of the item when d is its first slice)
            auto load_k = [&](const SD& d, uint32_t st, uint32_t bar) -> bool {
                if (x == 0 && (d.meta & 2u)) {
                    const uint32_t qs = (d.meta >> 3) & 1u, ph = (d.meta >> 4) & 1u;
                    if (!mbar_wait(q_empty(qs), ph ^ 1u, abort_flag, 11, P.status, P.wait_limit_ns)) return false;
                    mbar_expect_tx(q_full(qs), kBlockBytes);
                    tma_load_2d(sQ + qs * kBlockBytes, &P.map_q, d.qcol, d.qrow, q_full(qs));
                }
                tma_load_2d(sKx + st * kSliceB, &P.map_k, d.kcol, d.row, bar);
                return true;
            };
            auto load_v = [&](const SD& d, uint32_t st, uint32_t bar) {
                tma_load_2d(sVx + st * kSliceB, &P.map_v, d.vcol, d.row, bar);
            };
            // S_x of slice d (its K slice in stage st) into score buffer buf
            auto scores = [&](const SD& d, uint32_t st, uint32_t buf) -> bool {
                const uint32_t qs = (d.meta >> 3) & 1u;
                if (!(d.meta & 1u)) return true;
                if (d.meta & 2u) {
                    if (!mbar_wait(q_full(qs), (d.meta >> 4) & 1u, abort_flag, 12, P.status, P.wait_limit_ns)) return false;
                    tc_fence_after();
                }
                const uint64_t dq = dq0 + qs * (kBlockBytes >> 4), dk = dk0 + st * (kSliceB >> 4);
                const uint32_t ksteps = (d.meta >> 5) & 7u, t = tS + 64 * buf;
                tc_mma_bf16(t, dq, dk, idesc_s, 0u);
                if (ksteps > 1) tc_mma_bf16(t, dq + 2, dk + 2, idesc_s, 1u);
                if (ksteps > 2) tc_mma_bf16(t, dq + 4, dk + 4, idesc_s, 1u);
                if (ksteps > 3) tc_mma_bf16(t, dq + 6, dk + 6, idesc_s, 1u);
                tc_commit(s_full(x, buf));
                if (d.meta & 4u) tc_commit(q_empty(qs));
                return true;
            };
            SD d0 = next(), d1 = next(), d2 = next(), d3;
            {   // start: K slices 0 and 1 and V slice 0, and their score products; then K slice 2, on a barrier of its own.  (Where
                // every item is one slice long - three items to a CTA, sequences of 129 to 192 positions -, slice 2 brings the third Q
                // tile, whose buffer is free only after slice 0's product.)
                const uint32_t nk = (d0.meta & 1u) + (d1.meta & 1u);
                if (nk) mbar_expect_tx(kv_full(x, 0), (nk + 1) * kSliceB);
                if (d0.meta & 1u) {
                    ok = load_k(d0, 0, kv_full(x, 0));
                    load_v(d0, 0, kv_full(x, 0));
                }
                if (ok && (d1.meta & 1u)) ok = load_k(d1, 1, kv_full(x, 0));
                if (ok && nk) ok = mbar_wait(kv_full(x, 0), 0u, abort_flag, 12, P.status, P.wait_limit_ns);
                tc_fence_after();
                ok = ok && scores(d0, 0, 0) && scores(d1, 1, 1);
                if (ok && (d2.meta & 1u)) {
                    mbar_expect_tx(k2_full(x), kSliceB);
                    ok = load_k(d2, 2, k2_full(x));
                }
            }
            uint32_t G = 0, st0 = 0;                // st0 = G % 3
            while (ok && (d0.meta & 1u)) {
                const uint32_t buf = G & 1u, ph = (G >> 1) & 1u;
                const uint32_t st1 = st0 == 2 ? 0 : st0 + 1, st2 = st1 == 2 ? 0 : st1 + 1;
                if (!(ok = mbar_wait(p_full(x, buf), ph, abort_flag, 12, P.status, P.wait_limit_ns))) break;
                if (G > 0 && !(ok = mbar_wait(kv_full(x, buf), ph, abort_flag, 12, P.status, P.wait_limit_ns))) break;
                if (G == 0 && (d2.meta & 1u) && !(ok = mbar_wait(k2_full(x), 0u, abort_flag, 12, P.status, P.wait_limit_ns))) break;
                tc_fence_after();
                {   // O_x += P_x V_x over the slice's 64 keys
                    const uint32_t idesc_o = make_idesc(kTile, ((d0.meta >> 8) & 15u) << 4, 0, 1);
                    const uint64_t dv = dv0 + st0 * (kSliceB >> 4);
                    const uint32_t tP = tS + 64 * buf;
                    tc_mma_bf16_ts(tO, tP, dv, idesc_o, (d0.meta & 2u) ? 0u : 1u);
                    tc_mma_bf16_ts(tO, tP + 8, dv + 128, idesc_o, 1u);
                    tc_mma_bf16_ts(tO, tP + 16, dv + 256, idesc_o, 1u);
                    tc_mma_bf16_ts(tO, tP + 24, dv + 384, idesc_o, 1u);
                    tc_commit(pv_done(x, buf));
                }
                if (!(ok = scores(d2, st2, buf))) break;      // slice G + 2
                d3 = next();                                   // slice G + 3
                {
                    const uint32_t nb = (d3.meta & 1u) + (d1.meta & 1u), bar = kv_full(x, buf ^ 1u);
                    if (nb) mbar_expect_tx(bar, nb * kSliceB);
                    if ((d3.meta & 1u) && !(ok = load_k(d3, st0, bar))) break;
                    if (d1.meta & 1u) load_v(d1, st1, bar);
                }
                d0 = d1;
                d1 = d2;
                d2 = d3;
                st0 = st1;
                ++G;
            }
            // The items without a visible key for this stream are the last ones of the CTA's list (what an item sees never grows
            // along it).  Their Q buffers are handed back one by one, each once it has been filled: a hand-back ahead of that
            // would count towards the phase of an earlier item, and with several of them the buffer's phases run away from the
            // loader, which then waits for good.
            for (uint32_t k = g_qi + 1 - g_skip; ok && k != g_qi + 1; ++k) {
                if (!(ok = mbar_wait(q_full(k & 1u), (k >> 1) & 1u, abort_flag, 12, P.status, P.wait_limit_ns))) break;
                mbar_arrive(q_empty(k & 1u));
            }
        }
    } else {
        // ------------------------------------------------------------------ softmax streams
        const uint32_t x = static_cast<uint32_t>(warp - NS) >> 2;
        const int row = (warp & 3) * 32 + lane;
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const uint32_t tS0 = t_lane + Cfg::col_s(x, 0), tO = t_lane + Cfg::col_o(x);
        constexpr int CH = 32, NC = 64 / CH;
        uint32_t cs = 0, mi = 0;             // slices of this stream so far, items
        bool ok = true, pending_b = false;
        const int64_t T = static_cast<int64_t>(P.batch) * P.seq;
        for (int it = dealt_item(0); ok && it < P.n_items; it = dealt_item(++mi)) {
            const MsItem I = ms_decode(it, P.n_qt, P.n_heads, P.batch, P.seq, P.causal);
            const int n_own = ms_steps(I.lim, x, kKeys);
            const int wv = P.heads.vo_w[I.h];
            const int q_pos = I.qt * kTile + row;
            const int limit = P.causal ? min(P.seq, q_pos + 1) : P.seq;     // keys [0, limit) are visible
            RowState rsx;
            rsx.m = -1e30f;
            rsx.l = 0.f;
            for (int j = 0; j < n_own; ++j) {
                if (!(ok = mbar_wait(s_full(x, cs & 1), (cs >> 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
                tc_fence_after();
                const uint32_t tS = tS0 + 64 * (cs & 1), tP = tS;    // the probabilities go over the scores they came from
                const int kv_base = j * kKeys + 64 * static_cast<int>(x);
                const bool masked = kv_base + 64 > limit;                   // keys past the limit count as -inf
                float rs4[4] = {0.f, 0.f, 0.f, 0.f};
                uint32_t ra[CH], rb[CH];
                if constexpr (EXACT) {
                    // the slice's maximum before its exponentials: the reference is the stream's running maximum, so that the
                    // largest probability of a row is exactly 1 in the stream that has its key
                    tc_ld(tS, ra);
                    tc_ld(tS + CH, rb);
                    tc_wait_ld(ra);
                    tc_wait_ld(rb);
                    float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                    for (int i = 0; i < CH; ++i) {
                        if (masked && kv_base + i >= limit) ra[i] = 0xff800000u;
                        if (masked && kv_base + CH + i >= limit) rb[i] = 0xff800000u;
                    }
#pragma unroll
                    for (int i = 0; i < CH; i += 2) {
                        mx4[(i >> 1) & 1] = max3(mx4[(i >> 1) & 1], __uint_as_float(ra[i]), __uint_as_float(ra[i + 1]));
                        mx4[2 + ((i >> 1) & 1)] = max3(mx4[2 + ((i >> 1) & 1)], __uint_as_float(rb[i]), __uint_as_float(rb[i + 1]));
                    }
                    const float m_new = fmaxf(rsx.m, fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * P.scale_log2e);
                    const float f = ex2(rsx.m - m_new);
                    if (j > 0 && __any_sync(0xffffffffu, m_new > rsx.m)) {
                        if (!(ok = mbar_wait(pv_done(x, (cs - 1) & 1), ((cs - 1) >> 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
                        tc_fence_after();
                        for (int g = 0; g < (wv >> 4); ++g) {
                            uint32_t r[16];
                            tc_ld16(tO + 16 * g, r);
                            tc_wait_ld(r);
#pragma unroll
                            for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * f);
                            tc_st(tO + 16 * g, r);
                        }
                    }
                    rsx.m = m_new;
                    rsx.l *= f;
                    const f32x2 c2 = pack2(P.scale_log2e, P.scale_log2e), nm2 = pack2(-m_new, -m_new);
                    f32x2 acc2[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};
                    auto exponentiate = [&](const uint32_t (&v)[CH], uint32_t t) {
                        uint32_t pk[CH / 2];
#pragma unroll
                        for (int i = 0; i < CH; i += 2) {
                            float x0, x1;
                            unpack2(fma2(pack2(v[i], v[i + 1]), c2, nm2), x0, x1);
                            const float p0 = ex2(x0), p1 = ex2(x1);
                            acc2[(i >> 1) & 1] = add2(acc2[(i >> 1) & 1], pack2(p0, p1));
                            pk[i >> 1] = pack_bf16(p0, p1);
                        }
                        tc_st(t, pk);
                    };
                    exponentiate(ra, tP);
                    exponentiate(rb, tP + CH / 2);
                    unpack2(acc2[0], rs4[0], rs4[1]);
                    unpack2(acc2[1], rs4[2], rs4[3]);
                } else {
                    tc_ld(tS, ra);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        uint32_t(&cur)[CH] = (c & 1) ? rb : ra;
                        uint32_t(&nxt)[CH] = (c & 1) ? ra : rb;
                        tc_wait_ld(cur);
                        if (c + 1 < NC) tc_ld(tS + (c + 1) * CH, nxt);
                        if (masked) {
#pragma unroll
                            for (int i = 0; i < CH; ++i)
                                if (kv_base + c * CH + i >= limit) cur[i] = 0xff800000u;
                        }
                        // The chunk's maximum and its exponentials (with the reference the row has) have no dependence on one
                        // another, so they can be interleaved; only if some score exceeds the reference by more than 32 (rare) is
                        // the row rescaled and the chunk exponentiated again.
                        float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                        for (int i = 0; i < CH; i += 2) mx4[(i >> 1) & 3] = max3(mx4[(i >> 1) & 3], __uint_as_float(cur[i]), __uint_as_float(cur[i + 1]));
                        const float cm = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * P.scale_log2e;
                        uint32_t pk[CH / 2];
                        float cs4[4] = {0.f, 0.f, 0.f, 0.f};
                        auto exponentiate = [&](float neg_m) {   // (packed fp32 multiply-adds and sums: half the issue slots)
                            const f32x2 c2 = pack2(P.scale_log2e, P.scale_log2e), nm2 = pack2(neg_m, neg_m);
                            f32x2 acc2[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};
#pragma unroll
                            for (int i = 0; i < CH; i += 2) {
                                float x0, x1;
                                unpack2(fma2(pack2(cur[i], cur[i + 1]), c2, nm2), x0, x1);
                                const float p0 = ex2(x0), p1 = ex2(x1);
                                acc2[(i >> 1) & 1] = add2(acc2[(i >> 1) & 1], pack2(p0, p1));
                                pk[i >> 1] = pack_bf16(p0, p1);
                            }
                            unpack2(acc2[0], cs4[0], cs4[1]);
                            unpack2(acc2[1], cs4[2], cs4[3]);
                        };
                        exponentiate(-rsx.m);
                        if (__any_sync(0xffffffffu, cm - rsx.m > 32.f)) {
                            // the output row is touched: the product of the previous slice must have landed
                            if (j > 0 && !(ok = mbar_wait(pv_done(x, (cs - 1) & 1), ((cs - 1) >> 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
                            tc_fence_after();
                            rsx.rs = (rs4[0] + rs4[1]) + (rs4[2] + rs4[3]);
                            rsx = rescale_row(rsx, cm, tO, j > 0 ? wv >> 4 : 0, tP, c);
                            rs4[0] = rsx.rs;
                            rs4[1] = rs4[2] = rs4[3] = 0.f;
                            exponentiate(-rsx.m);
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q) rs4[q] += cs4[q];
                        tc_st(tP + c * (CH / 2), pk);
                    }
                }
                if (!ok) break;
                tc_wait_st();
                tc_fence_before();
                if (pending_b) {   // the output regions of the previous item have been read by every stream
                    if (!(ok = mbar_wait(merge_b, (mi - 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
                    pending_b = false;
                }
                mbar_arrive(p_full(x, cs & 1));
                rsx.l += (rs4[0] + rs4[1]) + (rs4[2] + rs4[3]);
                ++cs;
            }
            if (!ok) break;
            if (n_own > 0) {   // the stream's last product of the item
                if (!(ok = mbar_wait(pv_done(x, (cs - 1) & 1), ((cs - 1) >> 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
                tc_fence_after();
            }
            if (pending_b) {       // (a stream without slices in this item)
                if (!(ok = mbar_wait(merge_b, (mi - 1) & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
                pending_b = false;
            }
            // merge of the row's NS partial results
            merge[x * kTile + row] = rsx.m;
            merge[(NS + x) * kTile + row] = rsx.l;
            mbar_arrive(merge_a);
            if (!(ok = mbar_wait(merge_a, mi & 1u, abort_flag, 13, P.status, P.wait_limit_ns))) break;
            float gk[NS], M = -INFINITY, L = 0.f;
#pragma unroll
            for (int k = 0; k < NS; ++k)
                if (ms_steps(I.lim, k, kKeys) > 0) M = fmaxf(M, merge[k * kTile + row]);
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                gk[k] = 0.f;
                if (ms_steps(I.lim, k, kKeys) > 0) {
                    gk[k] = ex2(merge[k * kTile + row] - M);
                    L = fmaf(merge[(NS + k) * kTile + row], gk[k], L);
                }
            }
            const float inv = 1.f / L;
            const bool live = q_pos < P.seq;
            const int64_t t = static_cast<int64_t>(I.b) * P.seq + q_pos;
            for (int grp = x; grp < (wv >> 4); grp += NS) {   // this stream's share of the output columns
                float acc[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) acc[i] = 0.f;
#pragma unroll
                for (int k = 0; k < NS; ++k) {
                    if (ms_steps(I.lim, k, kKeys) > 0) {
                        uint32_t r[16];
                        tc_ld16(t_lane + Cfg::col_o(k) + 16 * grp, r);
                        tc_wait_ld(r);
#pragma unroll
                        for (int i = 0; i < 16; ++i) acc[i] = fmaf(__uint_as_float(r[i]), gk[k], acc[i]);
                    }
                }
                if (live) {
                    uint16_t* dst = P.ctx + t * P.ld_ctx + P.heads.vo_off[I.h] + 16 * grp;
                    uint4 v0, v1;
                    v0.x = pack_bf16(acc[0] * inv, acc[1] * inv);
                    v0.y = pack_bf16(acc[2] * inv, acc[3] * inv);
                    v0.z = pack_bf16(acc[4] * inv, acc[5] * inv);
                    v0.w = pack_bf16(acc[6] * inv, acc[7] * inv);
                    v1.x = pack_bf16(acc[8] * inv, acc[9] * inv);
                    v1.y = pack_bf16(acc[10] * inv, acc[11] * inv);
                    v1.z = pack_bf16(acc[12] * inv, acc[13] * inv);
                    v1.w = pack_bf16(acc[14] * inv, acc[15] * inv);
                    *reinterpret_cast<uint4*>(dst) = v0;
                    *reinterpret_cast<uint4*>(dst + 8) = v1;
                }
            }
            if (x == 0 && live) P.lse[static_cast<int64_t>(I.h) * T + t] = M * 0.6931471805599453f + logf(L);
            tc_fence_before();
            mbar_arrive(merge_b);
            pending_b = true;
        }
    }

    // ---------------------------------------------------------------------- teardown
    __syncwarp();
    if (*abort_flag) {
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);   // copies still in flight land before the memory is released
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// ------------------------------------------------------------------------------------------------
// backward
// ------------------------------------------------------------------------------------------------
// Reverse mode of Ctx_h = P V_h, P = softmax(scale * Q_h K_h^T), with P recomputed from the saved log-sum-exp:
//     dV = P^T dCtx,  dP = dCtx V^T,  dS = P (.) (dP - D),  D_t = sum_c dCtx[t, c] Ctx[t, c],
//     dQ = scale * dS K,  dK = scale * dS^T Q.
// Three launches: the row dots D with the log-sum-exp in the form the other two use (memory-bound), then one launch that
// owns key blocks (dK and dV accumulate in TMEM over the query blocks) and one that owns query blocks (dQ accumulates
// over the key blocks).  Nothing is added across CTAs, so the results do not depend on timing.

// A block takes kDotPos neighbouring positions of the padded sequences, a warp two of them at a time: every lane multiplies
// 16-byte vectors (8 columns, which never straddle a head because offsets and widths are multiples of 8), and the per-vector
// partial sums are added per head in order.  The row dots D_t = sum_c dCtx[t, c] Ctx[t, c] and the log-sum-exp in the form the
// backward kernels use are written in a layout whose 128-position blocks are whole, 512-byte aligned runs (so that a block's
// vectors can be copied to shared memory in bulk).  The head-major reads of the log-sum-exp and the
// writes go through whole 64-byte runs of positions.  (A warp per position touched a 32-byte sector for every 4-byte value;
// from the previous kernel's end to this one's 9.6 us at 8192 positions, 512 columns, launched on its own; now 5.7.)
constexpr int kDotWarps = 8, kDotPos = 2 * kDotWarps;
constexpr int kDotMaxVecs = 2048;      // 16384 columns
struct DotParams {
    HeadLayout heads;
    const uint16_t* ctx;
    const uint16_t* dctx;
    const float* lse;                  // [n_heads][T], natural logarithm (from the forward call)
    float* vecs;                       // [2][n_heads][batch][seq_pad]: -lse * log2(e), then the row dots D; zero past seq
    int64_t ld_ctx, ld_dctx, T;
    int32_t n_heads, n_vecs, batch, seq, seq_pad;
};
inline size_t dot_smem(int n_vecs, int n_heads) { return (static_cast<size_t>(kDotWarps) * 2 * n_vecs + static_cast<size_t>(n_heads) * (kDotPos + 1)) * 4; }
__device__ __forceinline__ float dot8(const uint4& x, const uint4& y) {
    float s = bf16_lo(x.x) * bf16_lo(y.x);
    s = fmaf(bf16_hi(x.x), bf16_hi(y.x), s);
    s = fmaf(bf16_lo(x.y), bf16_lo(y.y), s);
    s = fmaf(bf16_hi(x.y), bf16_hi(y.y), s);
    s = fmaf(bf16_lo(x.z), bf16_lo(y.z), s);
    s = fmaf(bf16_hi(x.z), bf16_hi(y.z), s);
    s = fmaf(bf16_lo(x.w), bf16_lo(y.w), s);
    return fmaf(bf16_hi(x.w), bf16_hi(y.w), s);
}
__global__ void __launch_bounds__(32 * kDotWarps) attn_rowdot_kernel(const __grid_constant__ DotParams P) {
    extern __shared__ float dot_smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* part = dot_smem_raw + warp * 2 * P.n_vecs;                 // [position][vector] of this warp
    float* dots = dot_smem_raw + kDotWarps * 2 * P.n_vecs;            // [head][kDotPos + 1]
    const int64_t tp = static_cast<int64_t>(blockIdx.x) * kDotPos;    // (whole blocks: the padded length is a multiple of 128)
    const int b = static_cast<int>(tp / P.seq_pad), pos0 = static_cast<int>(tp % P.seq_pad);
    pdl_start();
    pdl_wait();
    const int p0 = pos0 + 2 * warp;                                   // positions p0 and p0 + 1
    if (p0 < P.seq) {
        const int64_t t0 = static_cast<int64_t>(b) * P.seq + p0, t1 = static_cast<int64_t>(b) * P.seq + min(p0 + 1, P.seq - 1);
        const uint16_t* a0 = P.ctx + t0 * P.ld_ctx;
        const uint16_t* a1 = P.ctx + t1 * P.ld_ctx;
        const uint16_t* d0 = P.dctx + t0 * P.ld_dctx;
        const uint16_t* d1 = P.dctx + t1 * P.ld_dctx;
#pragma unroll 1
        for (int v = lane; v < P.n_vecs; v += 64) {                   // eight loads in flight
            const int v1 = min(v + 32, P.n_vecs - 1);                 // (past the end: the last vector again)
            const uint4 x0 = ld_stream16(a0 + 8 * v), y0 = ld_stream16(d0 + 8 * v), x1 = ld_stream16(a1 + 8 * v), y1 = ld_stream16(d1 + 8 * v);
            const uint4 x2 = ld_stream16(a0 + 8 * v1), y2 = ld_stream16(d0 + 8 * v1), x3 = ld_stream16(a1 + 8 * v1), y3 = ld_stream16(d1 + 8 * v1);
            part[v] = dot8(x0, y0);
            part[P.n_vecs + v] = dot8(x1, y1);
            if (v + 32 < P.n_vecs) {
                part[v + 32] = dot8(x2, y2);
                part[P.n_vecs + v + 32] = dot8(x3, y3);
            }
        }
        __syncwarp();
        for (int i = lane; i < 2 * P.n_heads; i += 32) {
            const int h = i >> 1, p = i & 1;
            const int v0 = P.heads.vo_off[h] >> 3, nv = P.heads.vo_w[h] >> 3;
            float s = 0.f;
            for (int k = 0; k < nv; ++k) s += part[p * P.n_vecs + v0 + k];
            dots[h * (kDotPos + 1) + 2 * warp + p] = s;
        }
    }
    __syncthreads();
    const int64_t per_arr = static_cast<int64_t>(P.n_heads) * P.batch * P.seq_pad;
    for (int i = threadIdx.x; i < P.n_heads * kDotPos; i += 32 * kDotWarps) {
        const int h = i / kDotPos, p = i % kDotPos, pos = pos0 + p;
        const int64_t o = (static_cast<int64_t>(h) * P.batch + b) * P.seq_pad + pos;
        const bool live = pos < P.seq;
        P.vecs[o] = live ? -P.lse[static_cast<int64_t>(h) * P.T + static_cast<int64_t>(b) * P.seq + pos] * 1.4426950408889634f : 0.f;
        P.vecs[per_arr + o] = live ? dots[h * (kDotPos + 1) + p] : 0.f;
    }
}

struct AttnBwdParams {
    alignas(64) CUtensorMap map_q, map_k, map_v, map_do;
    HeadLayout heads;
    int32_t batch, seq, n_heads, n_t, causal, n_items;
    float scale_log2e, scale;
    const float* vecs;                 // [2][n_heads][batch][seq_pad]: -lse * log2(e) and the row dots D (attn_rowdot_kernel)
    int32_t seq_pad;
    uint16_t* dq;
    uint16_t* dk;
    uint16_t* dv;
    int64_t ld_dqk, ld_dv;
    int* status;
    unsigned long long wait_limit_ns;
};

// MODE 0: a CTA owns a key block of a (sequence, K/V head) and walks the query blocks of the query heads that read it:
//         K, V resident, Q_i and dCtx_i streamed (with the step's queries' -lse*log2e and D, bulk-copied on the same
//         barrier); X = S^T = K Q_i^T and Y = dP^T = V dCtx_i^T (thread = key row, columns = queries); P^T and dS^T are
//         the A operands of dV += P^T dCtx_i and dK += dS^T Q_i, which accumulate in TMEM.
// MODE 1: a CTA owns a query block and walks the key blocks: Q, dCtx resident, K_j and V_j streamed; X = S = Q K_j^T and
//         Y = dP = dCtx V_j^T (thread = query row); dS is the A operand of dQ += dS K_j, which accumulates in TMEM.
// Streamed tiles serve twice: as K-major B operands of the score products and as MN-major B operands of the
// accumulating ones (same bytes, other descriptor).  A step is a streamed block of 64 rows.  Warp 0 loads, warps 2..17 compute, in
// two groups of eight that take the steps in turn, each with score tiles and packed operands of its own: while one waits
// for its products the other keeps the exponential unit busy.  What a step costs is a chain of short waits (scores, TMEM loads,
// exponentials, operands, products), not a pipe: the exponentials of 128 x 128 scores take 1024 clocks, a pair of steps 2200.
// Before (all warps on one block of 128, or on half blocks in turn) / now, us: 109 / 63 (60 x 48 positions, 32 heads 64
// wide), 134 / 112 (4 x 1000, 32 heads 48 wide on 8), 45.1 / 36.3 (32 x 197, 6 heads 48 wide, no mask), 106.5 / 100 (8 x 1024, 16
// heads 32 wide), 1045 / 969 (2 x 4096, 32 heads 128 wide).  Slower than before: heads up to 32 wide, two tiles, no mask, many items (54.0 /
// 58.3 for 512 heads of 256 positions, 35.2 / 37.2 for 256; causal 58.1 / 54.5).
// The products are issued by separate threads.  Heads up to 64 wide (NB = 1): warp 1 issues the score products; warps 18 and 19
// the accumulating ones (dV and dK; the query-block kernel needs only the second), whose A operands go through TMEM as
// packed bf16 beside the scores.  Wider heads (NB = 2): warp 1 issues X, warp 18 Y, warp 19 the accumulating products.  The
// accumulators of the key-block kernel then leave no TMEM columns beside the score tiles: every thread writes its packed P^T and
// dS^T over the scores it has made them from, and the buffer is free for the next scores when the products that read the
// operands are done.  On heads up to 64 wide the query-block kernel adds the products of even and of odd steps up in accumulators
// of their own, which are added at the end: a sum in one accumulator would be twice as long (and 0.3 us per item shorter to write
// out: 109.3 against 112.7 us at 4 x 1000, 32 heads 48 wide on 8, 98.3 against 99.4 at 8 x 1024, 16 heads 32 wide).
// Wait codes: 14 / 15 / 16 (MODE 0 loads, products, compute) and 17 / 18 / 19 (MODE 1).
constexpr int kStep = 64;                  // rows of a streamed block (queries in the key-block kernel, keys in the query-block kernel)
template <int NB, int MODE>
struct BwdCfg {
    static constexpr int kTileBytes = NB * kBlockBytes;
    static constexpr int kStrBlockBytes = kStep * 128;                         // 64 columns of a streamed block
    static constexpr int kStrTileBytes = NB * kStrBlockBytes;
    static constexpr int kResStages = NB == 1 ? 2 : 1;                         // buffers of the resident pair of tiles
    static constexpr int kStrStages = NB == 1 ? 6 : 4;                         // stages of the streamed pair of tiles
    static constexpr bool kOverlay = NB == 2 && MODE == 0;                      // operands over the scores
    static constexpr int kVecBytes = MODE == 0 ? kStrStages * 2 * kStep * 4 : 0;   // -lse2 and D of a query block, per streamed stage
    static constexpr int kSmem = 2 * kTileBytes * kResStages + 2 * kStrTileBytes * kStrStages + kVecBytes + 1024 + 512;
    static_assert(kSmem <= 232448, "shared memory of a block");
};

// NACC: accumulators.  Key-block kernel: 2 = those of two items side by side (heads at most 32 wide).  Query-block kernel: 3 or 4 (heads
// at most 64 or 32 wide) that the halves of the items' sums take in turn, 64 or 32 columns each; 2 = one for every other item, for
// sequences of one step (60 x 48, 32 heads, both kernels: 64.6 us instead of 68.6 on heads 64 wide, 59.1 instead of 64.5 on 48).
template <int NB, int MODE, int NACC = 1>
__global__ void __launch_bounds__(kBwdThreads, 1) attn_bwd_kernel(const __grid_constant__ AttnBwdParams P) {
    using Cfg = BwdCfg<NB, MODE>;
    constexpr int kTileBytes = Cfg::kTileBytes, kStrTileBytes = Cfg::kStrTileBytes, kStrBlockBytes = Cfg::kStrBlockBytes;
    constexpr int RS = Cfg::kResStages, SS = Cfg::kStrStages;
    // TMEM columns: two buffers of the score tiles X and Y, accumulators, two buffers of the packed bf16 operands of the
    // accumulating products (P^T and dS^T, or dS), two values per column
    constexpr uint32_t kAccIssuers = NB == 1 && MODE == 0 ? 2 : 1, kScoreIssuers = NB == 1 ? 1 : 2;
    constexpr uint32_t kColX = 0, kColY = 128, kColAcc = 256;
    // accumulator `which` (0: dV, 1: dK) of set as, or accumulator as of the query-block kernel
    auto col_acc = [](int which, uint32_t as) -> uint32_t {
        if (MODE == 1) return kColAcc + (NACC == 4 ? 32 : 64) * as;
        return kColAcc + (NACC == 2 ? 64 * as + 32 * which : (NB == 1 ? 64 : 128) * which);
    };
    // operand `which` (0: P^T, 1: dS^T or dS) of 16 contraction steps from 16 ks on, in operand buffer ob.  (Over the scores a
    // thread's 32 columns become its first 16.)
    auto col_op = [](int which, uint32_t ob, uint32_t ks) -> uint32_t {
        if (Cfg::kOverlay) return (which == 0 ? kColX : kColY) + 64 * ob + 32 * (ks >> 1) + 8 * (ks & 1);
        return (MODE == 0 ? 384 + 64 * which : 448) + 32 * ob + 8 * ks;
    };
    constexpr int kCodeBase = MODE == 0 ? 14 : 17;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (base - raw_addr);
    // resident: [stage][a | b], streamed: [stage][a | b], vectors, barriers
    const uint32_t sRes = base, sStr = sRes + 2 * kTileBytes * RS;
    uint8_t* vec_raw = smem + 2 * kTileBytes * RS + 2 * kStrTileBytes * SS;
    float* vec = reinterpret_cast<float*>(vec_raw);                               // [stage][-lse2 | D][kStep]
    uint8_t* tail = vec_raw + Cfg::kVecBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(tail);
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(tail + 32 * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 32 * 8 + 8);
    const uint32_t bar0 = smem_u32(bars);
    auto r_full = [&](uint32_t s) { return bar0 + 8u * s; };
    auto r_empty = [&](uint32_t s) { return bar0 + 8u * (2 + s); };
    auto t_full = [&](uint32_t s) { return bar0 + 8u * (4 + s); };
    auto t_empty = [&](uint32_t s) { return bar0 + 8u * (10 + s); };
    // per group of compute warps: scores complete; scores in registers; operands written; operands read
    auto x_full = [&](uint32_t b) { return bar0 + 8u * (16 + b); };
    auto xy_free = [&](uint32_t b) { return bar0 + 8u * (18 + b); };
    auto out_full = [&](uint32_t b) { return bar0 + 8u * (20 + b); };
    auto out_empty = [&](uint32_t b) { return bar0 + 8u * (22 + b); };
    // accumulators: one set, or several that the items (or the halves of their sums) take in turn, each with its own pair of barriers
    auto acc_full = [&](uint32_t a) { return bar0 + 8u * (24 + a); };
    auto acc_empty = [&](uint32_t a) { return bar0 + 8u * (28 + a); };
    constexpr uint32_t n_acc = NACC;
    constexpr bool kHalfSums = MODE == 1 && NACC > 2;             // sum 2 ri + (step & 1) of the item number ri, in accumulator (2 ri + (step & 1)) % n_acc
    static_assert(NB == 1 ? NACC <= 4 && (MODE == 1 || NACC <= 2) : NACC == 1, "several accumulators need the narrow layout");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < 2; ++s) {
            mbar_init(r_full(s), 1);
            mbar_init(r_empty(s), kScoreIssuers);
        }
        for (uint32_t s = 0; s < SS; ++s) {
            mbar_init(t_full(s), 1);
            mbar_init(t_empty(s), kAccIssuers);
        }
        for (uint32_t b = 0; b < 2; ++b) {
            mbar_init(x_full(b), kScoreIssuers);
            mbar_init(xy_free(b), kBwdComputeWarps / 2);  // barriers the compute threads arrive on: one arrival per warp (its lanes meet first)
            mbar_init(out_full(b), kBwdComputeWarps / 2);
            mbar_init(out_empty(b), kAccIssuers);
        }
        for (uint32_t a = 0; a < 4; ++a) {
            mbar_init(acc_full(a), kAccIssuers);
            mbar_init(acc_empty(a), kBwdComputeWarps);
        }
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tensormap(&P.map_q);
        prefetch_tensormap(&P.map_k);
        prefetch_tensormap(&P.map_v);
        prefetch_tensormap(&P.map_do);
    }
    pdl_start();
    if (warp == 1) tmem_alloc(smem_u32(tmem_holder), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    pdl_wait();

    // item -> (sequence, head, owned block, steps, first streamed block).  MODE 0 owns a key block of a K/V head and
    // walks the query blocks of every query head that reads it, one head after the other (h = the first of them).
    struct BItem {
        int b, h, own, n_steps, n_per, first;
    };
    const int grp = MODE == 0 ? P.heads.rep : 1;
    auto decode = [&](int it) {
        BItem I;
        const int per = (P.n_heads / grp) * P.batch;
        const int a = it / per;
        I.own = MODE == 0 ? a : P.n_t - 1 - a;                 // causal: the blocks with the most steps first
        const int rem = it % per;
        I.h = (rem / P.batch) * grp;
        I.b = rem % P.batch;
        if (MODE == 0) {
            I.first = P.causal ? I.own * (kTile / kStep) : 0;  // query blocks (of kStep queries) at or after the key block
            I.n_per = (P.seq + kStep - 1) / kStep - I.first;
        } else {
            I.first = 0;
            I.n_per = (P.seq + kStep - 1) / kStep;             // key blocks (of kStep keys) up to the end of the query block
            if (P.causal) I.n_per = min(I.n_per, (I.own + 1) * (kTile / kStep));
        }
        I.n_steps = I.n_per * grp;
        return I;
    };
    // which tensor maps / head columns the resident and streamed "a" (Q/K side) and "b" (V/dCtx side) tiles use
    const CUtensorMap* map_ra = MODE == 0 ? &P.map_k : &P.map_q;
    const CUtensorMap* map_rb = MODE == 0 ? &P.map_v : &P.map_do;
    const CUtensorMap* map_sa = MODE == 0 ? &P.map_q : &P.map_k;
    const CUtensorMap* map_sb = MODE == 0 ? &P.map_do : &P.map_v;

    // The score products X = Ra Sa^T (contraction over the Q/K width) and / or Y = Rb Sb^T (over the V width) of every step:
    // those of a step as soon as every compute thread has the previous scores of the same buffer in registers (it says so
    // half way through its step), also across the boundary between two items.
    auto score_role = [&](bool do_x, bool do_y) {
        uint32_t g = 0, ri = 0;
        bool ok = true;
        for (int it = dealt_item(0); ok && it < P.n_items; it = dealt_item(++ri)) {
            const BItem I = decode(it);
            const int wa = P.heads.qk_w[I.h], wb = P.heads.vo_w[I.h];
            const uint32_t rs = ri % RS;
            if (!(ok = mbar_wait(r_full(rs), (ri / RS) & 1u, abort_flag, kCodeBase + 1, P.status, P.wait_limit_ns))) break;
            const uint32_t idesc_x = make_idesc(kTile, kStep, 0, 0);
            const uint64_t d_ra = make_smem_desc(sRes + (2 * rs) * kTileBytes, 16, 1024),
                           d_rb = make_smem_desc(sRes + (2 * rs + 1) * kTileBytes, 16, 1024);
            for (int i = 0; ok && i < I.n_steps; ++i, ++g) {
                const uint32_t use = g >> 1, st = g % SS, xb = g & 1;
                if (use > 0 && !(ok = mbar_wait(Cfg::kOverlay ? out_empty(xb) : xy_free(xb), (use - 1) & 1u, abort_flag, kCodeBase + 1, P.status, P.wait_limit_ns))) break;
                if (!(ok = mbar_wait(t_full(st), (g / SS) & 1u, abort_flag, kCodeBase + 1, P.status, P.wait_limit_ns))) break;
                tc_fence_after();
                const uint64_t d_sa = make_smem_desc(sStr + (2 * st) * kStrTileBytes, 16, 1024),
                               d_sb = make_smem_desc(sStr + (2 * st + 1) * kStrTileBytes, 16, 1024);
                if (do_x) {
#pragma unroll
                    for (int ks = 0; ks < 4 * NB; ++ks) {
                        const uint32_t o = ((ks >> 2) * kBlockBytes + (ks & 3) * 32) >> 4, os = ((ks >> 2) * kStrBlockBytes + (ks & 3) * 32) >> 4;
                        if (ks < (wa >> 4)) tc_mma_bf16(tmem_base + kColX + xb * kStep, d_ra + o, d_sa + os, idesc_x, ks != 0 ? 1u : 0u);
                    }
                }
                if (do_y) {
#pragma unroll
                    for (int ks = 0; ks < 4 * NB; ++ks) {
                        const uint32_t o = ((ks >> 2) * kBlockBytes + (ks & 3) * 32) >> 4, os = ((ks >> 2) * kStrBlockBytes + (ks & 3) * 32) >> 4;
                        if (ks < (wb >> 4)) tc_mma_bf16(tmem_base + kColY + xb * kStep, d_rb + o, d_sb + os, idesc_x, ks != 0 ? 1u : 0u);
                    }
                }
                tc_commit(x_full(xb));
            }
            if (ok) tc_commit(r_empty(rs));
        }
    };
    // The accumulating products number w0 .. w1 - 1 of every step.  Key-block kernel: 0 is dV += P^T dCtx_i (B = streamed b
    // tile), 1 is dK += dS^T Q_i (B = streamed a tile); query-block kernel: 1 is dQ += dS K_j (B = streamed a tile), on heads up to
    // 64 wide in two sums, over the even and over the odd steps.
    auto acc_role = [&](int w0, int w1) {
        uint32_t g = 0, ri = 0;
        bool ok = true;
        for (int it = dealt_item(0); ok && it < P.n_items; it = dealt_item(++ri)) {
            const BItem I = decode(it);
            auto wait_acc = [&](uint32_t n) -> bool {                // the accumulator that takes sum number n has been written out
                return mbar_wait(acc_empty(n % n_acc), ((n / n_acc) & 1u) ^ 1u, abort_flag, kCodeBase + 1, P.status, P.wait_limit_ns);
            };
            for (int i = 0; i < I.n_steps; ++i, ++g) {
                const uint32_t st = g % SS, ob = g & 1, n = kHalfSums ? 2 * ri + (i & 1) : ri, as = n % n_acc;
                const int i_sum = kHalfSums ? i >> 1 : i;             // step of its sum
                if (!(ok = mbar_wait(t_full(st), (g / SS) & 1u, abort_flag, kCodeBase + 1, P.status, P.wait_limit_ns))) break;
                if (!(ok = mbar_wait(out_full(ob), (g >> 1) & 1u, abort_flag, kCodeBase + 1, P.status, P.wait_limit_ns))) break;
                if (i_sum == 0 && !(ok = wait_acc(n))) break;
                tc_fence_after();
                for (int which = w0; which < w1; ++which) {
                    const int wn = which == 0 ? P.heads.vo_w[I.h] : P.heads.qk_w[I.h];
                    const uint32_t idesc = make_idesc(kTile, wn, 0, 1);
                    const uint32_t acc = tmem_base + col_acc(MODE == 0 ? which : 0, as), op = tmem_base + col_op(which, ob, 0);
                    const uint64_t db = make_smem_desc(sStr + (2 * st + (which == 0 ? 1 : 0)) * kStrTileBytes, kStrBlockBytes, 1024);
#pragma unroll
                    for (int ks = 0; ks < kStep / 16; ++ks)
                        tc_mma_bf16_ts(acc, op + (Cfg::kOverlay ? 32 * (ks >> 1) + 8 * (ks & 1) : 8 * ks), db + 128 * ks, idesc, (i_sum | ks) != 0 ? 1u : 0u);
                }
                tc_commit(out_empty(ob));
                tc_commit(t_empty(st));
            }
            if (kHalfSums) {                                         // (one step: the second sum is empty, its turn is taken all the same)
                if (ok && I.n_steps == 1) ok = wait_acc(2 * ri + 1);
                if (ok) {
                    tc_commit(acc_full((2 * ri) % n_acc));
                    tc_commit(acc_full((2 * ri + 1) % n_acc));
                }
            } else if (ok) {
                tc_commit(acc_full(ri % n_acc));
            }
        }
    };

    if (warp == 0) {
        // ------------------------------------------------------------------ producer
        if (elect_one()) {
            uint32_t g = 0, ri = 0;
            bool ok = true;
            for (int it = dealt_item(0); ok && it < P.n_items; it = dealt_item(++ri)) {
                const BItem I = decode(it);
                // columns of the resident tiles: MODE 0 the K/V head's block of K^c and V^c, MODE 1 the query head's of Q^c and dCtx
                const int ra_off = MODE == 0 ? P.heads.k_off[I.h] : P.heads.qk_off[I.h];
                const int rb_off = MODE == 0 ? P.heads.v_off[I.h] : P.heads.vo_off[I.h];
                const int nba = (P.heads.qk_w[I.h] + 63) >> 6, nbb = (P.heads.vo_w[I.h] + 63) >> 6;
                const int row0 = I.b * P.seq;
                const uint32_t rs = ri % RS;
                if (!(ok = mbar_wait(r_empty(rs), ((ri / RS) & 1u) ^ 1u, abort_flag, kCodeBase, P.status, P.wait_limit_ns))) break;
                mbar_expect_tx(r_full(rs), (nba + nbb) * kBlockBytes);
                for (int half = 0; half < 2; ++half) {              // (all boxes are 64 rows high)
                    const uint32_t dst = sRes + (2 * rs) * kTileBytes + half * kStep * 128;
                    const int y = row0 + I.own * kTile + half * kStep;
                    for (int blk = 0; blk < nba; ++blk) tma_load_2d(dst + blk * kBlockBytes, map_ra, ra_off + 64 * blk, y, r_full(rs));
                    for (int blk = 0; blk < nbb; ++blk) tma_load_2d(dst + kTileBytes + blk * kBlockBytes, map_rb, rb_off + 64 * blk, y, r_full(rs));
                }
                for (int i = 0; i < I.n_steps; ++i, ++g) {
                    const uint32_t st = g % SS;
                    if (!(ok = mbar_wait(t_empty(st), ((g / SS) & 1u) ^ 1u, abort_flag, kCodeBase, P.status, P.wait_limit_ns))) break;
                    mbar_expect_tx(t_full(st), (nba + nbb) * kStrBlockBytes + (MODE == 0 ? 2 * kStep * 4 : 0));
                    // streamed tiles: MODE 0 the query block of query head h + i / n_per, MODE 1 the key block of the K/V head
                    const int hq = I.h + i / I.n_per;
                    if (MODE == 0) {   // with the query block's per-query vectors
                        const int64_t o = (static_cast<int64_t>(hq) * P.batch + I.b) * P.seq_pad + (I.first + i % I.n_per) * kStep;
                        const int64_t per_arr = static_cast<int64_t>(P.n_heads) * P.batch * P.seq_pad;
                        const uint32_t dst = smem_u32(vec) + st * 2 * kStep * 4;
                        bulk_load(dst, P.vecs + o, kStep * 4, t_full(st));
                        bulk_load(dst + kStep * 4, P.vecs + per_arr + o, kStep * 4, t_full(st));
                    }
                    const int sa_off = MODE == 0 ? P.heads.qk_off[hq] : P.heads.k_off[I.h];
                    const int sb_off = MODE == 0 ? P.heads.vo_off[hq] : P.heads.v_off[I.h];
                    const int y = row0 + (I.first + i % I.n_per) * kStep;
                    for (int blk = 0; blk < nba; ++blk)
                        tma_load_2d(sStr + (2 * st) * kStrTileBytes + blk * kStrBlockBytes, map_sa, sa_off + 64 * blk, y, t_full(st));
                    for (int blk = 0; blk < nbb; ++blk)
                        tma_load_2d(sStr + (2 * st + 1) * kStrTileBytes + blk * kStrBlockBytes, map_sb, sb_off + 64 * blk, y, t_full(st));
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ issuer of the score products
        if (elect_one()) score_role(true, NB == 1);
    } else if (warp >= 2 + kBwdComputeWarps) {
        // ------------------------------------------------------------------ issuers of the accumulating products (wide heads: of Y, and of all accumulating products)
        if (elect_one()) {
            const int which = warp - (2 + kBwdComputeWarps);
            if (MODE == 0 && NB == 1) acc_role(which, which + 1);
            else if (which == 1) acc_role(MODE, 2);
            else if (NB == 2) score_role(false, true);
        }
    } else {
        // ------------------------------------------------------------------ compute
        // Two groups of eight warps take the steps in turn (group = score buffer); thread = (row of the owned block = TMEM lane, half
        // of the streamed block's 64 columns), so every scheduler has two warps of each group.
        const int part = (warp - 2) >> 2, group = part >> 1;
        const int row = (warp & 3) * 32 + lane;
        constexpr int kHalves = 2;                                     // 16-column halves of this thread's columns
        const int col0 = (part & 1) * 32;                              // this thread's columns of the streamed block
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        uint32_t g = 0, ri = 0;
        bool ok = true;
        struct Pend {
            int h, b, own;
            uint32_t ri;
            bool on, two;                                              // two: both halves of the sum have products
        };
        Pend pend = {0, 0, 0, 0, false, false};
        // writes an item's accumulators out once they are complete (every thread a quarter of the columns) and releases them.  On heads
        // of 33 to 64 columns the later quarters are the smaller ones: dK, and the dQ of every second item, go out with the quarters
        // exchanged between the two groups, so that it is not always the same one that is held up (111.7 against 113.9 us at 16 x 1024,
        // 8 heads 48 wide, 67.5 against 69.3 at 64 x 256 without a mask; heads of at most 32, 4 x 2048: 314 against 307, wider ones the same).
        constexpr bool kExchange = NB == 1 && NACC == (MODE == 0 ? 1 : 3);
        auto flush = [&](const Pend& d) -> bool {
            const uint32_t n = kHalfSums ? 2 * d.ri : d.ri, as = n % n_acc, as2 = (n + 1) % n_acc;   // (as2: the second half's)
            if (!mbar_wait(acc_full(as), (n / n_acc) & 1u, abort_flag, kCodeBase + 2, P.status, P.wait_limit_ns)) return false;
            if (kHalfSums && !mbar_wait(acc_full(as2), ((n + 1) / n_acc) & 1u, abort_flag, kCodeBase + 2, P.status, P.wait_limit_ns)) return false;
            tc_fence_after();
            const int pos = d.own * kTile + row;
            const bool live = pos < P.seq;
            const int64_t t = static_cast<int64_t>(d.b) * P.seq + pos;
            auto write_acc = [&](uint32_t colbase, int quarter, int w, uint16_t* dst, float mul) {
#pragma unroll
                for (int c = 0; c < NB; ++c) {
                    const int col = quarter * (NB * 16) + c * 16;
                    if (col < w) {
                        uint32_t r[16];
                        tc_ld16(t_lane + colbase + col, r);
                        if (kHalfSums && d.two) {
                            uint32_t r2[16];
                            tc_ld16(t_lane + col_acc(0, as2) + col, r2);
                            tc_wait_ld(r2);
                            tc_wait_ld(r);
#pragma unroll
                            for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) + __uint_as_float(r2[e]));
                        } else {
                            tc_wait_ld(r);
                        }
                        if (live) {
                            uint4 v0, v1;
                            v0.x = pack_bf16(__uint_as_float(r[0]) * mul, __uint_as_float(r[1]) * mul);
                            v0.y = pack_bf16(__uint_as_float(r[2]) * mul, __uint_as_float(r[3]) * mul);
                            v0.z = pack_bf16(__uint_as_float(r[4]) * mul, __uint_as_float(r[5]) * mul);
                            v0.w = pack_bf16(__uint_as_float(r[6]) * mul, __uint_as_float(r[7]) * mul);
                            v1.x = pack_bf16(__uint_as_float(r[8]) * mul, __uint_as_float(r[9]) * mul);
                            v1.y = pack_bf16(__uint_as_float(r[10]) * mul, __uint_as_float(r[11]) * mul);
                            v1.z = pack_bf16(__uint_as_float(r[12]) * mul, __uint_as_float(r[13]) * mul);
                            v1.w = pack_bf16(__uint_as_float(r[14]) * mul, __uint_as_float(r[15]) * mul);
                            *reinterpret_cast<uint4*>(dst + col) = v0;
                            *reinterpret_cast<uint4*>(dst + col + 8) = v1;
                        }
                    }
                }
            };
            if (MODE == 0) {
                write_acc(col_acc(0, as), part, P.heads.vo_w[d.h], P.dv + t * P.ld_dv + P.heads.v_off[d.h], 1.f);
                write_acc(col_acc(1, as), kExchange ? part ^ 2 : part, P.heads.qk_w[d.h], P.dk + t * P.ld_dqk + P.heads.k_off[d.h], P.scale);
            } else {
                write_acc(col_acc(0, as), kExchange ? part ^ (2 * (d.ri & 1)) : part, P.heads.qk_w[d.h], P.dq + t * P.ld_dqk + P.heads.qk_off[d.h], P.scale);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(acc_empty(as));
                if (kHalfSums) mbar_arrive(acc_empty(as2));
            }
            return true;
        };
        for (int it = dealt_item(0); ok && it < P.n_items; it = dealt_item(++ri)) {
            const BItem I = decode(it);
            const int own_pos = I.own * kTile + row;                 // position of this thread's row in the sequence
            // MODE 1: this row's -log-sum-exp (base 2) and row dot (zeros past the end of the sequence).  MODE 0: the values of
            // the step's 64 queries arrive in shared memory with the step's tiles.
            float lse_r = 0.f, d_r = 0.f;
            if (MODE == 1) {
                const int64_t o = (static_cast<int64_t>(I.h) * P.batch + I.b) * P.seq_pad + own_pos;
                lse_r = P.vecs[o];
                d_r = P.vecs[static_cast<int64_t>(P.n_heads) * P.batch * P.seq_pad + o];
            }
            const int i0 = (g & 1) == static_cast<uint32_t>(group) ? 0 : 1;
            const uint32_t g_next = g + I.n_steps;
            g += i0;
            int blk = i0;                                            // step i of its query head (MODE 0: the heads of a group follow one another)
            for (int i = i0; i < I.n_steps; i += 2, g += 2, blk += 2) {
                while (MODE == 0 && blk >= I.n_per) blk -= I.n_per;
                const int other0 = (I.first + blk) * kStep;          // first position of the streamed block
                const float* vb = vec + (g % SS) * 2 * kStep;
                const uint32_t xb = g & 1, ob = xb;
                // (the step's loads landed long ago; this thread reads the vectors among them, so it looks at their barrier itself)
                if (MODE == 0 && !(ok = mbar_wait(t_full(g % SS), (g / SS) & 1u, abort_flag, kCodeBase + 2, P.status, P.wait_limit_ns))) break;
                if (!(ok = mbar_wait(x_full(xb), (g >> 1) & 1u, abort_flag, kCodeBase + 2, P.status, P.wait_limit_ns))) break;
                tc_fence_after();
                // (query position, key position) of element (row, column c): MODE 0 rows are keys, MODE 1 rows are queries
                const int q0 = MODE == 0 ? other0 : I.own * kTile, k0 = MODE == 0 ? I.own * kTile : other0;
                const bool masked = q0 + (MODE == 0 ? kStep : kTile) > P.seq || k0 + (MODE == 0 ? kTile : kStep) > P.seq ||
                                    (P.causal && q0 < k0 + (MODE == 0 ? kTile : kStep));
                // this thread's visible columns (MODE 0: queries at or after the row's key, MODE 1: keys up to the row's query)
                const int vis_lo = MODE == 0 && P.causal ? own_pos - q0 - col0 : 0;
                const int vis_hi = own_pos >= P.seq ? 0 : (MODE == 1 && P.causal ? min(P.seq, own_pos + 1) : P.seq) - other0 - col0;
                // two halves of 16 columns: probabilities and dS are packed to bf16 pairs as soon as they exist
                uint32_t pk_p[8 * kHalves], pk_ds[8 * kHalves];
                const f32x2 c2 = pack2(P.scale_log2e, P.scale_log2e), neg1 = pack2(-1.f, -1.f);
#pragma unroll
                for (int hh = 0; hh < kHalves; ++hh) {
                    uint32_t rx[16], ry[16];
                    tc_ld16(t_lane + kColX + xb * kStep + col0 + 16 * hh, rx);
                    tc_ld16(t_lane + kColY + xb * kStep + col0 + 16 * hh, ry);
                    tc_wait_ld();
                    if (!Cfg::kOverlay && hh == kHalves - 1) {        // this thread's last read of the step's score tiles
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(xy_free(xb));
                    }
                    if (masked) {                                     // pairs outside the mask count as -inf (p = 0)
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            if (16 * hh + e < vis_lo || 16 * hh + e >= vis_hi) rx[e] = 0xff800000u;
                    }
#pragma unroll
                    for (int e = 0; e < 16; e += 4) {
                        // packed fp32 arithmetic around the exponentials: the step is bound by issue slots as much as by the
                        // exponential unit.  l2 = -lse * log2(e); p = 2^(s * c + l2); dS = p * (dP - D)
                        f32x2 l2a = pack2(lse_r, lse_r), l2b = l2a, dda = pack2(d_r, d_r), ddb = dda;
                        if (MODE == 0) {
                            const float4 a4 = *reinterpret_cast<const float4*>(vb + col0 + 16 * hh + e);
                            const float4 b4 = *reinterpret_cast<const float4*>(vb + kStep + col0 + 16 * hh + e);
                            l2a = pack2(a4.x, a4.y); l2b = pack2(a4.z, a4.w);
                            dda = pack2(b4.x, b4.y); ddb = pack2(b4.z, b4.w);
                        }
                        float x0, x1, x2, x3;
                        unpack2(fma2(pack2(rx[e], rx[e + 1]), c2, l2a), x0, x1);
                        unpack2(fma2(pack2(rx[e + 2], rx[e + 3]), c2, l2b), x2, x3);
                        const float p0 = ex2(x0), p1 = ex2(x1), p2 = ex2(x2), p3 = ex2(x3);
                        float d0, d1, d2, d3;
                        unpack2(mul2(pack2(p0, p1), fma2(dda, neg1, pack2(ry[e], ry[e + 1]))), d0, d1);
                        unpack2(mul2(pack2(p2, p3), fma2(ddb, neg1, pack2(ry[e + 2], ry[e + 3]))), d2, d3);
                        pk_p[8 * hh + (e >> 1)] = pack_bf16(p0, p1);
                        pk_p[8 * hh + (e >> 1) + 1] = pack_bf16(p2, p3);
                        pk_ds[8 * hh + (e >> 1)] = pack_bf16(d0, d1);
                        pk_ds[8 * hh + (e >> 1) + 1] = pack_bf16(d2, d3);
                    }
                }
                // the products that read the operands last in this buffer are done (over the scores: the score products waited for that)
                if (!Cfg::kOverlay && !(ok = mbar_wait(out_empty(ob), ((g >> 1) & 1u) ^ 1u, abort_flag, kCodeBase + 2, P.status, P.wait_limit_ns))) break;
                // this thread's columns, packed, in its TMEM lane
                if (MODE == 0) tc_st(t_lane + col_op(0, ob, (part & 1) * kHalves), pk_p);
                tc_st(t_lane + col_op(1, ob, (part & 1) * kHalves), pk_ds);
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(out_full(ob));
                if (pend.on) {   // the previous item's accumulators, now that this item's first step is on its way
                    if (!(ok = flush(pend))) break;
                    pend.on = false;
                }
            }
            if (!ok) break;
            if (pend.on && !(ok = flush(pend))) break;         // (an item without a step for this group)
            g = g_next;
            pend = {I.h, I.b, I.own, ri, true, I.n_steps > 1};                // written out after the first step of the next item, when the last products into them have long landed
        }
        if (ok && pend.on) flush(pend);
    }

    // ---------------------------------------------------------------------- teardown
    __syncwarp();
    if (*abort_flag) {
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                              const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn attn_encode_fn() {
    static EncodeFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeFn>(p);
    });
    return fn;
}
// bf16 row-major (rows x cols, pitch ld) as tiles of 64 columns x box_rows rows, 128-byte swizzle, zero fill outside
ecospa_status_t encode_tile_map(CUtensorMap* out, const void* ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows = kTile) {
    EncodeFn enc = attn_encode_fn();
    if (!enc) {
        set_cuda_error(cudaErrorNotSupported, "cuTensorMapEncodeTiled entry point");
        return ECOSPA_ERR_CUDA;
    }
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld) * 2};
    const cuuint32_t box[2] = {64, static_cast<cuuint32_t>(box_rows)};
    const cuuint32_t estr[2] = {1, 1};
    if (enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
        set_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled (attention)");
        return ECOSPA_ERR_CUDA;
    }
    return ECOSPA_OK;
}

// Host-only checks shared by the forward and the backward call; fills the layout and the widths of the tensors: Q^c
// (n_qk), Ctx (n_vo), K^c (n_k) and V^c (n_v; the last two equal the first two unless K/V heads are shared).
ecospa_status_t check_heads(const ecospa_heads_t* heads, HeadLayout& L, int64_t& n_qk, int64_t& n_vo, int64_t& n_k, int64_t& n_v,
                            int& max_w) {
    if (!heads || !heads->qk_off || !heads->qk_w || !heads->vo_off || !heads->vo_w) return ECOSPA_ERR_INVALID;
    if (heads->n_heads < 1 || heads->n_kv_heads < 0) return ECOSPA_ERR_INVALID;
    if (heads->n_heads > kMaxHeads) return ECOSPA_ERR_UNSUPPORTED;
    const int n_kv = heads->n_kv_heads;
    if (n_kv > 0 && (!heads->k_off || !heads->v_off || heads->n_heads % n_kv != 0)) return ECOSPA_ERR_INVALID;
    const int rep = n_kv > 0 ? heads->n_heads / n_kv : 1;
    L.rep = rep;
    n_qk = n_vo = n_k = n_v = 0;
    max_w = 0;
    for (int h = 0; h < heads->n_heads; ++h) {
        const int32_t qo = heads->qk_off[h], qw = heads->qk_w[h], vo = heads->vo_off[h], vw = heads->vo_w[h];
        const int32_t ko = n_kv > 0 ? heads->k_off[h / rep] : qo, vko = n_kv > 0 ? heads->v_off[h / rep] : vo;
        if (qo < 0 || vo < 0 || ko < 0 || vko < 0 || qw < 1 || vw < 1) return ECOSPA_ERR_INVALID;
        if (qw > 128 || vw > 128) return ECOSPA_ERR_UNSUPPORTED;
        if ((qw & 15) || (vw & 15) || (qo & 7) || (vo & 7) || (ko & 7) || (vko & 7)) return ECOSPA_ERR_ALIGNMENT;
        // the query heads of a group share the group's kept indices, hence its widths
        if (h % rep != 0 && (qw != heads->qk_w[h - h % rep] || vw != heads->vo_w[h - h % rep])) return ECOSPA_ERR_INVALID;
        L.qk_off[h] = qo; L.qk_w[h] = qw; L.vo_off[h] = vo; L.vo_w[h] = vw; L.k_off[h] = ko; L.v_off[h] = vko;
        n_qk = std::max<int64_t>(n_qk, qo + qw);
        n_vo = std::max<int64_t>(n_vo, vo + vw);
        n_k = std::max<int64_t>(n_k, ko + qw);
        n_v = std::max<int64_t>(n_v, vko + vw);
        max_w = std::max(max_w, std::max(qw, vw));
    }
    return ECOSPA_OK;
}
ecospa_status_t check_mat(const void* p, int64_t ld, int64_t cols) {
    if (!p || ld < cols) return ECOSPA_ERR_INVALID;
    if (!aligned16(p) || (ld * 2) % 16) return ECOSPA_ERR_ALIGNMENT;
    return ECOSPA_OK;
}

}  // namespace

}  // namespace ecospa

using namespace ecospa;

extern "C" ecospa_status_t ecospa_coupled_attn_fwd(const void* Qc, const void* Kc, int64_t ld_qk, const void* Vc, int64_t ld_v,
                                                   int64_t batch, int64_t seq, const ecospa_heads_t* heads, float scale,
                                                   int32_t causal, void* Ctx, int64_t ld_ctx, float* lse, void* stream) {
    static thread_local AttnFwdParams P;
    int64_t n_qk = 0, n_vo = 0, n_k = 0, n_v = 0;
    int max_w = 0;
    ecospa_status_t st = check_heads(heads, P.heads, n_qk, n_vo, n_k, n_v, max_w);
    if (st != ECOSPA_OK) return st;
    if (batch < 1 || seq < 1 || batch * seq > INT32_MAX || !lse) return ECOSPA_ERR_INVALID;
    if (!(scale > 0.f) || !std::isfinite(scale)) return ECOSPA_ERR_INVALID;
    if ((st = check_mat(Qc, ld_qk, n_qk)) != ECOSPA_OK || (st = check_mat(Kc, ld_qk, n_k)) != ECOSPA_OK ||
        (st = check_mat(Vc, ld_v, n_v)) != ECOSPA_OK || (st = check_mat(Ctx, ld_ctx, n_vo)) != ECOSPA_OK)
        return st;
    if (reinterpret_cast<uintptr_t>(lse) & 3u) return ECOSPA_ERR_ALIGNMENT;
    int* status = engine_status_ptr(&st);
    if (!status) return st;
    const int64_t T = batch * seq;
    P.batch = static_cast<int32_t>(batch);
    P.seq = static_cast<int32_t>(seq);
    P.n_heads = heads->n_heads;
    P.n_qt = static_cast<int32_t>(ceil_div(seq, kTile));
    P.causal = causal != 0;
    const int64_t units = static_cast<int64_t>(P.n_heads) * batch, sms = std::max(1, engine_num_sms());
    // Few query tiles: one per SM (2 x 160 positions, 12 heads: 10.4 -> 8.1 us)
    P.items = units * P.n_qt <= sms ? ITEMS_SINGLE : P.n_qt == 1 ? ITEMS_SOLO : ITEMS_SHARED;
    // (Causal sequences of up to two tiles: 200 positions, 80 wide, 63 us without turns, 67 with; 768: 93 and 90.)
    P.turns = P.items == ITEMS_SHARED && (!P.causal || P.n_qt > 2);
    const int64_t tile_items = P.items == ITEMS_SINGLE ? units * P.n_qt : P.items == ITEMS_SOLO ? (units + 1) / 2 : units * ((P.n_qt + 1) / 2);
    // Output heads up to 32 wide (and Q/K heads up to 64): the kernel of key streams (K / V tiles as slices of 64 keys), but for
    // many short sequences; everything else: the kernel of tiles, with one or two 64-column blocks per tile.  The width is a
    // line of precision: the stream kernel rounds a row's probabilities to bf16 against a reference up to 2^32 below the row's
    // largest, the other kernel against the largest itself, which is then exactly 1.  On rows that few keys dominate (scores of
    // deviation 4, 1000 positions, 64 wide) the outputs are 1.7e-3 off the values in 64 bits, all of it their own rounding;
    // streams for the wider heads too were 2.3e-3 off.  Up to two tiles the streams take exact maxima too (one or two slices each, so
    // that the second look at the scores costs up to 0.6 us of 6.7): 1.74e-3 off there on such rows, the tile kernel 1.77e-3, streams without
    // exact maxima 1.95e-3 (72 heads of 256 positions, 32 wide, causal).  The length is one of time, in rounds of items over the SMs: an item of the
    // stream kernel is a query tile, one of the tile kernel up to two.  With sequences of one tile a round takes about as long in
    // both, with two tiles half as long again in the tile kernel; longer ones are always faster as streams.  Streams / tiles, us, 8
    // heads 32 wide, no mask and causal: 5.5 / 6.0, 5.5 / 6.0 (16 units of 128 positions), 5.8 / 6.6, 5.8 / 6.7 (144), 9.3 / 7.3, 9.5 / 7.4
    // (200), 11.9 / 9.8, 12.3 / 10.2 (320); 7.3 / 7.5, 7.3 / 7.6 (16 of 256), 7.4 / 8.2, 7.3 / 8.2 (72), 11.8 / 9.9, 9.4 / 9.2 (96), 15.8 / 15.4, 14.4 /
    // 14.9 (200), 23.9 / 20.6, 22.5 / 19.2 (320); 13.2 / 13.8, 12.3 / 13.7 (200 of 160); 16 heads, 8192 positions, causal: 34.2 / 36.2 (sequences of 512), 44.8 / 51 (1024).
    int max_vo = 0;
    for (int h = 0; h < heads->n_heads; ++h) max_vo = std::max<int>(max_vo, heads->vo_w[h]);
    const int64_t stream_rounds = ceil_div(units * P.n_qt, sms), tile_rounds = ceil_div(tile_items, sms);
    const bool streams = max_w <= 64 && max_vo <= 32 && (P.n_qt > 2 || (P.n_qt == 2 ? 2 * stream_rounds <= 3 * tile_rounds : stream_rounds <= tile_rounds));
    if ((st = encode_tile_map(&P.map_q, Qc, T, n_qk, ld_qk)) != ECOSPA_OK) return st;
    if ((st = encode_tile_map(&P.map_k, Kc, T, n_k, ld_qk, streams ? 64 : kTile)) != ECOSPA_OK) return st;
    if ((st = encode_tile_map(&P.map_v, Vc, T, n_v, ld_v, streams ? 64 : kTile)) != ECOSPA_OK) return st;
    const int64_t items = streams ? units * P.n_qt : tile_items;
    if (items > INT32_MAX) return ECOSPA_ERR_UNSUPPORTED;
    P.n_items = static_cast<int32_t>(items);
    P.scale_log2e = scale * 1.4426950408889634f;
    P.ctx = static_cast<uint16_t*>(Ctx);
    P.ld_ctx = ld_ctx;
    P.lse = lse;
    P.status = status;
    P.wait_limit_ns = engine_wait_limit_ns();
    static std::once_flag once[64];
    int dev = 0;
    cudaGetDevice(&dev);
    cudaError_t e = cudaSuccess;
    std::call_once(once[dev & 63], [&] {
        e = cudaFuncSetAttribute(attn_fwd_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdCfg<1>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_fwd_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdCfg<1>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_fwd_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdCfg<2>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_fwd_kernel<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdCfg<2>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_fwd_ms_kernel<3, 32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, MsCfg<3, 32>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_fwd_ms_kernel<3, 32, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, MsCfg<3, 32>::kSmem);
    });
    if (e != cudaSuccess) {
        set_cuda_error(e, "attention setup");
        cudaGetLastError();
        return ECOSPA_ERR_CUDA;
    }
    const int grid = std::min<int>(P.n_items, std::max(1, engine_num_sms()));
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    if (streams) return launch_pdl(P.n_qt <= 2 ? attn_fwd_ms_kernel<3, 32, true> : attn_fwd_ms_kernel<3, 32, false>, grid, MsCfg<3, 32>::kThreads, cs, P, "attn_fwd_kernel", MsCfg<3, 32>::kSmem);
    // Output rows through shared memory: stored straight from the threads, each with a row of its own, 64 columns of both streams take
    // 2400 to 2900 clocks, which nothing hides at the end of a CTA's last items (and all end together without a mask); items of one
    // key block, and causal ones on heads up to 64, rather wait for the longer way.  Direct / through shared memory, us: no mask 10.9 / 10.4 (96
    // heads of 256 positions, 64 wide), 17.4 / 16.1 (192 of 197, ragged), 26.0 / 24.9 (128 of 512), 12.5 / 11.2 (96 of 256, 96 wide), 166.5 / 164.3 (64
    // of 2048); causal 17.4 / 16.5 (72 of 512, 96 wide), 91.8 / 90.2 (64 of 2048), 16.4 / 17.0 (256 of 200, 80 wide), 20.4 / 20.8 (128 of 512, 64
    // wide); one key block 26.7 / 28.3 (1920 of 48, 48 wide), 8.7 / 9.2 (320 of 64, 32 wide).
    const bool staged = P.items != ITEMS_SOLO && (!P.causal || max_w > 64);
    if (max_w <= 64) return launch_pdl(staged ? attn_fwd_kernel<1, true> : attn_fwd_kernel<1, false>, grid, kFwdThreads, cs, P, "attn_fwd_kernel", FwdCfg<1>::kSmem);
    return launch_pdl(staged ? attn_fwd_kernel<2, true> : attn_fwd_kernel<2, false>, grid, kFwdThreads, cs, P, "attn_fwd_kernel", FwdCfg<2>::kSmem);
}

extern "C" size_t ecospa_attn_workspace_bytes(int64_t batch, int64_t seq, int32_t n_heads) {
    if (batch < 1 || seq < 1 || n_heads < 1) return 0;
    // two fp32 per (head, position of the sequences padded to whole blocks of 128): -lse * log2(e) and the row dots D
    return static_cast<size_t>(batch) * ceil_div(seq, static_cast<int64_t>(kTile)) * kTile * n_heads * 8 + 256;
}

extern "C" ecospa_status_t ecospa_coupled_attn_bwd(const void* Qc, const void* Kc, int64_t ld_qk, const void* Vc, int64_t ld_v,
                                                   const void* Ctx, int64_t ld_ctx, const void* dCtx, int64_t ld_dctx,
                                                   const float* lse, int64_t batch, int64_t seq, const ecospa_heads_t* heads,
                                                   float scale, int32_t causal, void* dQc, void* dKc, int64_t ld_dqk,
                                                   void* dVc, int64_t ld_dv, void* workspace, size_t workspace_bytes,
                                                   void* stream_) {
    static thread_local AttnBwdParams P;
    static thread_local DotParams D;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int64_t n_qk = 0, n_vo = 0, n_k = 0, n_v = 0;
    int max_w = 0;
    ecospa_status_t st = check_heads(heads, P.heads, n_qk, n_vo, n_k, n_v, max_w);
    if (st != ECOSPA_OK) return st;
    if (batch < 1 || seq < 1 || batch * seq > INT32_MAX || !lse) return ECOSPA_ERR_INVALID;
    if (!(scale > 0.f) || !std::isfinite(scale)) return ECOSPA_ERR_INVALID;
    if ((st = check_mat(Qc, ld_qk, n_qk)) != ECOSPA_OK || (st = check_mat(Kc, ld_qk, n_k)) != ECOSPA_OK ||
        (st = check_mat(Vc, ld_v, n_v)) != ECOSPA_OK || (st = check_mat(Ctx, ld_ctx, n_vo)) != ECOSPA_OK ||
        (st = check_mat(dCtx, ld_dctx, n_vo)) != ECOSPA_OK || (st = check_mat(dQc, ld_dqk, n_qk)) != ECOSPA_OK ||
        (st = check_mat(dKc, ld_dqk, n_k)) != ECOSPA_OK || (st = check_mat(dVc, ld_dv, n_v)) != ECOSPA_OK)
        return st;
    if (reinterpret_cast<uintptr_t>(lse) & 3u) return ECOSPA_ERR_ALIGNMENT;
    if (n_vo / 8 > kDotMaxVecs) return ECOSPA_ERR_UNSUPPORTED;
    if (!workspace || workspace_bytes < ecospa_attn_workspace_bytes(batch, seq, heads->n_heads)) return ECOSPA_ERR_WORKSPACE;
    if (!aligned16(workspace)) return ECOSPA_ERR_ALIGNMENT;
    int* status = engine_status_ptr(&st);
    if (!status) return st;
    const int64_t T = batch * seq;
    if ((st = encode_tile_map(&P.map_q, Qc, T, n_qk, ld_qk, kStep)) != ECOSPA_OK) return st;
    if ((st = encode_tile_map(&P.map_k, Kc, T, n_k, ld_qk, kStep)) != ECOSPA_OK) return st;
    if ((st = encode_tile_map(&P.map_v, Vc, T, n_v, ld_v, kStep)) != ECOSPA_OK) return st;
    if ((st = encode_tile_map(&P.map_do, dCtx, T, n_vo, ld_dctx, kStep)) != ECOSPA_OK) return st;
    float* vecs = static_cast<float*>(workspace);
    P.batch = static_cast<int32_t>(batch);
    P.seq = static_cast<int32_t>(seq);
    P.n_heads = heads->n_heads;
    P.n_t = static_cast<int32_t>(ceil_div(seq, kTile));
    P.causal = causal != 0;
    const int64_t items = static_cast<int64_t>(P.n_t) * P.n_heads * batch;
    if (items > INT32_MAX) return ECOSPA_ERR_UNSUPPORTED;
    P.n_items = static_cast<int32_t>(items);
    P.scale = scale;
    P.scale_log2e = scale * 1.4426950408889634f;
    P.vecs = vecs;
    P.seq_pad = static_cast<int32_t>(ceil_div(seq, static_cast<int64_t>(kTile)) * kTile);
    P.dq = static_cast<uint16_t*>(dQc);
    P.dk = static_cast<uint16_t*>(dKc);
    P.dv = static_cast<uint16_t*>(dVc);
    P.ld_dqk = ld_dqk;
    P.ld_dv = ld_dv;
    P.status = status;
    P.wait_limit_ns = engine_wait_limit_ns();
    static std::once_flag once[64];
    int dev = 0;
    cudaGetDevice(&dev);
    cudaError_t e = cudaSuccess;
    std::call_once(once[dev & 63], [&] {
        e = cudaFuncSetAttribute(attn_bwd_kernel<1, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdCfg<1, 0>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_bwd_kernel<1, 0, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdCfg<1, 0>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_bwd_kernel<1, 1, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdCfg<1, 1>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_bwd_kernel<1, 1, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdCfg<1, 1>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_bwd_kernel<1, 1, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdCfg<1, 1>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_bwd_kernel<2, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdCfg<2, 0>::kSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_bwd_kernel<2, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdCfg<2, 1>::kSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(attn_rowdot_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(dot_smem(kDotMaxVecs, kMaxHeads)));
    });
    if (e != cudaSuccess) {
        set_cuda_error(e, "attention backward setup");
        cudaGetLastError();
        return ECOSPA_ERR_CUDA;
    }
    // row dots D
    D.heads = P.heads;
    D.ctx = static_cast<const uint16_t*>(Ctx);
    D.dctx = static_cast<const uint16_t*>(dCtx);
    D.vecs = vecs;
    D.lse = lse;
    D.batch = static_cast<int32_t>(batch);
    D.seq = static_cast<int32_t>(seq);
    D.seq_pad = P.seq_pad;
    D.ld_ctx = ld_ctx;
    D.ld_dctx = ld_dctx;
    D.T = T;
    D.n_heads = heads->n_heads;
    D.n_vecs = static_cast<int32_t>(n_vo / 8);
    if ((st = launch_pdl(attn_rowdot_kernel, static_cast<unsigned>(batch * D.seq_pad / kDotPos), 32 * kDotWarps, stream, D, "attn_rowdot_kernel",
                         dot_smem(D.n_vecs, D.n_heads))) != ECOSPA_OK)
        return st;
    const int nb = max_w > 64 ? 2 : 1;
    // dK, dV: one item per (sequence, K/V head, key block); dQ: one per (sequence, query head, query block)
    const int items_q = P.n_items;
    P.n_items = items_q / P.heads.rep;
    int grid = std::min<int>(P.n_items, std::max(1, engine_num_sms()));
    if (nb == 1)
        st = launch_pdl(max_w <= 32 ? attn_bwd_kernel<1, 0, 2> : attn_bwd_kernel<1, 0, 1>, grid, kBwdThreads, stream, P,
                        "attn_bwd_kernel (dK, dV)", BwdCfg<1, 0>::kSmem);
    else
        st = launch_pdl(attn_bwd_kernel<2, 0, 1>, grid, kBwdThreads, stream, P, "attn_bwd_kernel (dK, dV)", BwdCfg<2, 0>::kSmem);
    if (st != ECOSPA_OK) return st;
    P.n_items = items_q;
    grid = std::min<int>(P.n_items, std::max(1, engine_num_sms()));
    if (nb == 1)
        return launch_pdl(seq <= kStep ? attn_bwd_kernel<1, 1, 2> : max_w <= 32 ? attn_bwd_kernel<1, 1, 4> : attn_bwd_kernel<1, 1, 3>, grid, kBwdThreads, stream, P,
                          "attn_bwd_kernel (dQ)", BwdCfg<1, 1>::kSmem);
    return launch_pdl(attn_bwd_kernel<2, 1, 1>, grid, kBwdThreads, stream, P, "attn_bwd_kernel (dQ)", BwdCfg<2, 1>::kSmem);
}

// Grouped persistent bf16 GEMM for sm_100a: TMA -> shared memory ring -> tcgen05.mma (fp32 accumulators
// in TMEM, double buffered) -> fused epilogues.  Four forms of the same kernel:
//   slim    cta_group::1, one CTA per SM computes 128x64 tiles (4 stages of 2 x (16 KB A + 8 KB B)): launches that
//           such tiles cover in one round
//   single  the same with 128x128 tiles (3 stages of 2 x (16 KB A + 16 KB B)): launches that such tiles cover in one round
//   wide    the same with 128x256 tiles (2 stages of 2 x (16 KB A + 32 KB B)): longer launches of at most 128 rows, where
//           the second CTA of a pair would compute nothing
//   pair    cta_group::2, a cluster of two CTAs computes 256x256 tiles: each CTA loads its 128 rows of A
//           and its half of B (3 stages of 2 x (16 KB + 16 KB)), the leader CTA issues the MMAs for both,
//           so every SM fetches a third less operand data per flop.  Every CTA issues its own loads: the
//           peer's loads signal the leader's barrier, and completion is committed to each CTA's barrier.
//
// One launch computes up to kMaxGemmOps independent products ("ops"), each C = sum over one to three
// K segments of A_seg * B_seg with K-major or MN-major operands (chosen per segment, so that weights
// and activations are consumed in whatever row-major orientation they are stored).  Warp roles:
//   warp 0      producer: one elected lane issues the TMA loads of a stage (two 64-deep k-blocks)
//   warp 1      owns the 512 TMEM columns; one elected lane issues the MMAs and the commits
//   warps 2..9  epilogue: two warps per TMEM lane quadrant, each takes half of the tile's columns; a warp
//               converts its rows, stages them in swizzled shared memory and one lane issues a TMA tile
//               store (a reducing store when the output is added to what C holds)
// Tiles are numbered op by op, longest contraction first; the host hands them out longest first to the
// least-loaded worker and passes the lists as a table in the kernel parameters (a plain stride when
// there are many tiles per worker).  The kernel is launched with programmatic stream serialization and
// touches no global memory before griddepcontrol.wait, so its set-up overlaps the previous kernel's tail.
// Every mbarrier wait is bounded in time; on expiry the CTA records an error code in a device
// status word, waits for its copies in flight, frees its TMEM and returns.

#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "gemm.cuh"

namespace ecospa {

namespace {

constexpr int BM = 128, BK = 64;
constexpr int kAStage = BM * BK * 2;        // 16 KB: 128 rows of A
constexpr int kSub = 2;                     // 64-deep k-blocks per pipeline stage
constexpr int kMaxStages = 4;
constexpr int kRingBytes = 192 * 1024;
// Tile of a worker, by form: rows and columns, and the ring that brings its operands.
enum TileForm { TILE_SINGLE = 0, TILE_PAIR = 1, TILE_WIDE = 2, TILE_SLIM = 3 };
template <int FORM>
struct TileShape {
    static constexpr int kM = FORM == TILE_PAIR ? 2 * BM : BM, kN = FORM == TILE_SLIM ? 64 : FORM == TILE_SINGLE ? 128 : 256;
    static constexpr int kTmemCols = 2 * kN;               // two accumulators
    static constexpr int kBStage = (FORM == TILE_PAIR ? kN / 2 : kN) * BK * 2;   // B bytes of a CTA per k-block (a pair's holds half the tile's columns)
    static constexpr int kStages = FORM == TILE_WIDE ? 2 : FORM == TILE_SLIM ? 4 : 3;
    static_assert(kStages * kSub * (kAStage + kBStage) == kRingBytes, "ring of a CTA");
};
constexpr int kAtomBytes = 64 * 64 * 2;     // one 64x64 bf16 swizzle atom of an MN-major operand
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kMaxSeg = 3;
constexpr int kEpiSlotBytes = 32 * 32 * 2;  // one 32-row x 64-byte staging image; a warp owns two (= one 32 x 128-byte image)
constexpr int kEpiBytes = kEpiWarps * 2 * kEpiSlotBytes;
constexpr int kSmemBytes = kRingBytes + kEpiBytes + 1024 /*alignment slack*/ + 256 /*barriers*/;
constexpr unsigned long long kDefaultWaitLimitNs = 2000000000ull;  // 2 s

struct DevProblem {
    int32_t M, N;
    int32_t kb_end[kMaxSeg];     // cumulative k-blocks: segment s covers [kb_end[s-1], kb_end[s])
    int32_t kblocks;             // k-blocks of all segments
    int32_t tiles_m, tiles_n, tile_start;
    int32_t n_per_tile;          // output columns per tile: the tile's, or half as many hidden units for EPI_SWIGLU
    int32_t half1_n_off;         // n-coordinate of B half 1 relative to half 0
    int32_t epi;
    int32_t k_off[kMaxSeg];      // first contraction index of each segment
    uint8_t a_mn[kMaxSeg], b_mn[kMaxSeg];
    uint8_t map_a[kMaxSeg], map_b[kMaxSeg][2];
    uint8_t a_3d[kMaxSeg], b_3d[kMaxSeg];   // MN-major operand fetched as one 3-D box (both 64-wide atoms)
    uint8_t a_big[kMaxSeg], b_big[kMaxSeg]; // pair mode: one box brings both k-blocks of a stage
    uint8_t map_c[3];            // store maps of C, C2, C3
    uint8_t pad2_[2];
    uint8_t out_f32, accumulate, bias_f32, pad_[5];
    void* C;
    void* C2;
    void* C3;
    const void* bias;
    const void* H;
    const void* Hb;
    int64_t ldc, ldh;
};

constexpr uint16_t kNoTile = 0xffff;
struct GemmHead {
    // Worker w runs, in round i, tile order[w + i * workers] (kNoTile = nothing) when use_order is set,
    // otherwise tile w + i * workers.
    int32_t n_problems, total_tiles, rounds, use_order;
    int* status;
    unsigned long long wait_limit_ns;   // every mbarrier wait of the launch gives up after this long
    SideSums side;
};
// Kernel parameters in two sizes: what a launch costs the host grows with them (measured with an idle queue, a call of the
// score kernels with 29 KB took 43-79 us for three launches and takes 16 with 1.7 KB).  Most launches fit the small form (a call's operands, one map each); the large one is for
// weight gradients split over the tokens and for schedules of many tiles.
template <int MAPS, int OPS, int ORDER>
struct GemmParams {
    static constexpr int kMaps = MAPS, kOps = OPS, kOrder = ORDER;
    alignas(64) CUtensorMap maps[MAPS];
    DevProblem prob[OPS];
    GemmHead head;
    uint16_t order[ORDER];               // the explicit tile schedule
};
using LargeParams = GemmParams<72, kMaxGemmOps, 2048>;
using SmallParams = GemmParams<20, 5, 512>;

__device__ int g_gemm_status = 0;

// ------------------------------------------------------------------------------------------------
// PTX wrappers
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// True in one lane (always the same) of a converged warp.  The branches whose thread issues loads, stores and products are
// entered through this and not through a comparison of the lane number, because it measured faster (see tc.cuh; here, loads alone
// back behind a comparison: 15.8 -> 16.6 us for Q/K/V of 4096 rows, 1024 / 512, 7.4 -> 7.8 for 1024 rows).
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait.  Returns false if the wait gave up (or another thread of the CTA already did).
template <bool CLUSTER>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int code, int* status,
                                          unsigned long long limit_ns) {
    // Fast path: plain polling.  The (slow) global timer is only consulted every 1024 failed polls,
    // so a wait that completes normally never touches it (limits under a millisecond look at it on
    // every failed poll, so that they are kept to within a poll).
    unsigned long long t0 = 0;
    uint32_t spins = 0;
    const uint32_t mask = limit_ns < 1000000ull ? 0u : 1023u;
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((++spins & mask) == 0) {
            if (*abort_flag) return false;
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > limit_ns) {
                *abort_flag = 1;
                atomicCAS(status, 0, code);
                return false;
            }
        }
    }
}

// --- cluster (CTA pair) helpers
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// shared::cluster address of `addr` (a shared::cta address of this CTA) in the CTA of rank `rank`
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// TMA load issued by one CTA of a pair; the completion may be signalled on the peer's (leader's) barrier.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar_cluster) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar_cluster), "r"(x), "r"(y)
        : "memory");
}
__device__ __forceinline__ void tc_commit_pair(uint32_t bar_cluster) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar_cluster) : "memory");
}
__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int y, int z, int w, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(0), "r"(y), "r"(z), "r"(w)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap* map, int y, int z, int w, uint32_t bar_cluster) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar_cluster), "r"(0), "r"(y), "r"(z), "r"(w)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar_cluster) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar_cluster), "r"(x), "r"(y), "r"(z)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y)
        : "memory");
}

// --- TMA tile stores (shared memory -> global), tracked per issuing thread in bulk groups
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
}
// C += tile: the addition is done by the memory system in the output's type, once per element
__device__ __forceinline__ void tma_reduce_add_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
    asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// all but the newest N stores of this thread have finished reading their shared-memory source
template <int N>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32]) {
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
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((addr >> 4) & 0x3fffu);
    d |= static_cast<uint64_t>((lbo_bytes >> 4) & 0x3fffu) << 16;
    d |= static_cast<uint64_t>((sbo_bytes >> 4) & 0x3fffu) << 32;
    d |= 1ull << 46;   // descriptor version of this architecture
    d |= 2ull << 61;   // 128-byte swizzle
    return d;
}

// ------------------------------------------------------------------------------------------------
// epilogue math (fp32)
// ------------------------------------------------------------------------------------------------
// The erf-form GELU needs Phi(x), the standard normal CDF, for 32768 outputs per tile, which makes the
// epilogue ALU-bound if it is evaluated with exponentials and divisions.  Here
//   Phi(x) ~= 1/2 + xc * Q(xc^2),   xc = clamp(x, -4.5, 4.5),
// with Q a degree-8 polynomial fitted (weighted least squares on Chebyshev nodes, refitted towards the
// minimax error) to (Phi(x) - 1/2)/x on [0, 4.5]; |error| <= 2.1e-5 everywhere (the clamp contributes
// 3.4e-6), far below the bf16 rounding of the outputs.  Two elements are evaluated per instruction with
// the packed fp32 pair arithmetic of this architecture.
typedef unsigned long long f32x2;   // two fp32 values in one 64-bit register
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float ex2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Phi of two values
__device__ __forceinline__ f32x2 normal_cdf2(float x0, float x1) {
    const f32x2 xc = pack2(fminf(fmaxf(x0, -4.5f), 4.5f), fminf(fmaxf(x1, -4.5f), 4.5f));
    const f32x2 t = mul2(xc, xc);
    f32x2 q = pack2(3.80569048497037e-11f, 3.80569048497037e-11f);
    q = fma2(q, t, pack2(-4.0023149239232225e-09f, -4.0023149239232225e-09f));
    q = fma2(q, t, pack2(1.8461658157775673e-07f, 1.8461658157775673e-07f));
    q = fma2(q, t, pack2(-4.959736997989239e-06f, -4.959736997989239e-06f));
    q = fma2(q, t, pack2(8.72766540851444e-05f, 8.72766540851444e-05f));
    q = fma2(q, t, pack2(-0.0010767392814159393f, -0.0010767392814159393f));
    q = fma2(q, t, pack2(0.009729491546750069f, 0.009729491546750069f));
    q = fma2(q, t, pack2(-0.06624043732881546f, -0.06624043732881546f));
    q = fma2(q, t, pack2(0.3988664746284485f, 0.3988664746284485f));
    return fma2(xc, q, pack2(0.5f, 0.5f));
}
// v[i] <- GELU(v[i]) = v[i] Phi(v[i])
__device__ __forceinline__ void gelu_erf32(float (&v)[32]) {
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
        const f32x2 g = mul2(pack2(v[i], v[i + 1]), normal_cdf2(v[i], v[i + 1]));
        unpack2(g, v[i], v[i + 1]);
    }
}
// v[i] <- v[i] * GELU'(h[i]),  GELU'(h) = Phi(h) + h phi(h),  phi(h) = exp(-h^2/2)/sqrt(2 pi).
// With hc = clamp(h, -4.5, 4.5) and t = hc^2:  Phi ~= 1/2 + hc Q6(t) (degree-6 fit of the same kind as above,
// |error| <= 3.0e-4, an order of magnitude below the bf16 rounding of the result) and
// phi = 2^(-t log2(e)/2 - log2(sqrt(2 pi))); beyond the clamp both terms are within 1e-4 of their limits.
__device__ __forceinline__ void dgelu_erf32(float (&v)[32], const float (&h)[32]) {
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
        const f32x2 hc = pack2(fminf(fmaxf(h[i], -4.5f), 4.5f), fminf(fmaxf(h[i + 1], -4.5f), 4.5f));
        const f32x2 t = mul2(hc, hc);
        const f32x2 ex = fma2(t, pack2(-0.72134752044448170f, -0.72134752044448170f),
                              pack2(-1.3257480647361593f, -1.3257480647361593f));
        float e0, e1;
        unpack2(ex, e0, e1);
        f32x2 q = pack2(1.431838114740458e-08f, 1.431838114740458e-08f);
        q = fma2(q, t, pack2(-1.1645848871921771e-06f, -1.1645848871921771e-06f));
        q = fma2(q, t, pack2(3.9588092477060854e-05f, 3.9588092477060854e-05f));
        q = fma2(q, t, pack2(-0.0007395460270345211f, -0.0007395460270345211f));
        q = fma2(q, t, pack2(0.008474125526845455f, 0.008474125526845455f));
        q = fma2(q, t, pack2(-0.06415736675262451f, -0.06415736675262451f));
        q = fma2(q, t, pack2(0.39786770939826965f, 0.39786770939826965f));
        // Phi + h phi = 1/2 + hc (Q6 + phi)
        const f32x2 qp = add2(pack2(ex2_fast(e0), ex2_fast(e1)), q);
        const f32x2 d = fma2(hc, qp, pack2(0.5f, 0.5f));
        const f32x2 r = mul2(pack2(v[i], v[i + 1]), d);
        unpack2(r, v[i], v[i + 1]);
    }
}
// tanh(u) = 1 - 2 / (1 + exp(2u)); saturates correctly for large |u|
__device__ __forceinline__ float tanh_fast(float u) { return 1.f - __fdividef(2.f, 1.f + __expf(2.f * u)); }
__device__ __forceinline__ float gelu_tanh(float x) {
    const float u = 0.79788456080286536f * (x + 0.044715f * x * x * x);
    return 0.5f * x * (1.f + tanh_fast(u));
}
__device__ __forceinline__ float dgelu_tanh(float x) {
    const float u = 0.79788456080286536f * (x + 0.044715f * x * x * x);
    const float t = tanh_fast(u);
    const float du = 0.79788456080286536f * (1.f + 3.f * 0.044715f * x * x);
    return 0.5f * (1.f + t) + 0.5f * x * (1.f - t * t) * du;
}
__device__ __forceinline__ float sigmoidf_(float x) { return __fdividef(1.f, 1.f + __expf(-x)); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// Staging images for the TMA tile stores.  A warp owns 4 KB: either one image of 32 rows x 128 bytes in the
// 128-byte swizzle (64 bf16 or 32 fp32 columns; 16-byte chunk j of row r sits at chunk j ^ (r & 7)), or two
// "slots" of 32 rows x 64 bytes in the 64-byte swizzle (32 bf16 columns; chunk j of row r at j ^ ((r >> 1) & 3)).
// Lane = row (what tcgen05.ld delivers); both layouts are bank-conflict free for that access.
// Before an image is overwritten the issuing lane waits until the stores that still read it are done
// (KEEP = stores that may stay in flight because they read the other slot).
template <int KEEP>
__device__ __forceinline__ void stage_begin(int lane) {
    bulk_wait_read<KEEP>();                // (nothing to wait for in the lanes that issued none)
    __syncwarp();
}
__device__ __forceinline__ void stage_commit(const CUtensorMap* map, uint32_t buf, int x, int y, int lane, bool add = false) {
    fence_async_smem();
    __syncwarp();
    if (elect_one()) {
        if (add) tma_reduce_add_2d(map, buf, x, y);
        else tma_store_2d(map, buf, x, y);
        bulk_commit();
    }
}
// 32 words (128 bytes) per lane
__device__ __forceinline__ void stage_row128(uint32_t buf, int lane, const uint32_t (&w)[32]) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(buf + lane * 128 + ((j ^ (lane & 7)) << 4)),
                     "r"(w[4 * j]), "r"(w[4 * j + 1]), "r"(w[4 * j + 2]), "r"(w[4 * j + 3]) : "memory");
}
// 64 fp32 values of one row -> 64 bf16 columns (one 128-byte image row)
__device__ __forceinline__ void stage_bf16x64(uint32_t buf, int lane, const float (&v0)[32], const float (&v1)[32]) {
    uint32_t w[32];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        w[i] = pack_bf16(v0[2 * i], v0[2 * i + 1]);
        w[16 + i] = pack_bf16(v1[2 * i], v1[2 * i + 1]);
    }
    stage_row128(buf, lane, w);
}
// 32 fp32 values of one row -> 32 fp32 columns (one 128-byte image row)
__device__ __forceinline__ void stage_f32x32(uint32_t buf, int lane, const float (&v)[32]) {
    uint32_t w[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) w[i] = __float_as_uint(v[i]);
    stage_row128(buf, lane, w);
}
// 32 fp32 values of one row -> 32 bf16 columns (one 64-byte slot row)
__device__ __forceinline__ void stage_bf16x32(uint32_t slot, int lane, const float (&v)[32]) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(slot + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4)),
                     "r"(pack_bf16(v[8 * c + 0], v[8 * c + 1])), "r"(pack_bf16(v[8 * c + 2], v[8 * c + 3])),
                     "r"(pack_bf16(v[8 * c + 4], v[8 * c + 5])), "r"(pack_bf16(v[8 * c + 6], v[8 * c + 7]))
                     : "memory");
}

// Landing buffer of the saved activations: 32 rows x 32 bf16 columns, 64 bytes per row, the four 16-byte
// chunks of a row permuted by (chunk ^ ((row >> 1) & 3)) so that both access patterns are conflict-free:
//   "line" pattern: 4 lanes per row, 8 rows per instruction (coalesced 64-byte global segments);
//   "row" pattern:  lane = row, a lane touches the four chunks of its row (the layout of tcgen05.ld).
__device__ __forceinline__ uint32_t epi_chunk_addr(uint32_t buf, int row, int chunk) {
    return buf + row * 64 + ((chunk ^ ((row >> 1) & 3)) << 4);
}

// global (bf16, rows m_warp.. x columns n..n+31) -> registers in the coalesced "line" pattern.  Split in
// two so that the global loads of the next chunk are in flight while the current one is processed.
__device__ __forceinline__ void staged_load32_issue(const unsigned short* H, int64_t ldh, int m_warp, int n, int M, int N,
                                                    uint4 (&q)[4], int lane) {
    const int c = lane & 3;
    const int col = n + 8 * c;
    if (m_warp + 32 <= M && n + 32 <= N) {      // the whole block is inside: four plain vector loads
        const unsigned short* g0 = H + static_cast<int64_t>(m_warp + (lane >> 2)) * ldh + col;
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = *reinterpret_cast<const uint4*>(g0 + static_cast<int64_t>(8 * i) * ldh);
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = 8 * i + (lane >> 2);
        q[i] = make_uint4(0, 0, 0, 0);
        if (m_warp + row < M && col < N) {
            const unsigned short* g = H + static_cast<int64_t>(m_warp + row) * ldh + col;
            if (col + 8 <= N) {
                q[i] = *reinterpret_cast<const uint4*>(g);
            } else {
                uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (col + e < N) w[e >> 1] |= static_cast<uint32_t>(g[e]) << ((e & 1) * 16);
                q[i] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    }
}
// registers ("line" pattern) -> buffer -> registers (one row per lane, fp32)
__device__ __forceinline__ void staged_load32_finish(uint32_t buf, const uint4 (&q)[4], float (&v)[32], int lane) {
    const int c = lane & 3;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = 8 * i + (lane >> 2);
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(epi_chunk_addr(buf, row, c)), "r"(q[i].x), "r"(q[i].y), "r"(q[i].z), "r"(q[i].w) : "memory");
    }
    __syncwarp();
#pragma unroll
    for (int cc = 0; cc < 4; ++cc) {
        uint4 t;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(t.x), "=r"(t.y), "=r"(t.z), "=r"(t.w) : "r"(epi_chunk_addr(buf, lane, cc)));
        v[8 * cc + 0] = bf16_lo(t.x); v[8 * cc + 1] = bf16_hi(t.x);
        v[8 * cc + 2] = bf16_lo(t.y); v[8 * cc + 3] = bf16_hi(t.y);
        v[8 * cc + 4] = bf16_lo(t.z); v[8 * cc + 5] = bf16_hi(t.z);
        v[8 * cc + 6] = bf16_lo(t.w); v[8 * cc + 7] = bf16_hi(t.w);
    }
    __syncwarp();
}

// tile of worker `worker` in round `i`, or -1
template <typename Params>
__device__ __forceinline__ int scheduled_tile(const Params& P, int worker, int n_workers, int i) {
    const int pos = worker + i * n_workers;
    if (P.head.use_order) {
        const int t = P.order[pos];
        return t == kNoTile ? -1 : t;
    }
    return pos < P.head.total_tiles ? pos : -1;
}

// v[i] += bias of column i, where lane i of the warp holds that column's bias
__device__ __forceinline__ void add_bias32(float (&v)[32], float b) {
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] += __shfl_sync(0xffffffffu, b, i);
}

template <typename Params>
__device__ __forceinline__ const DevProblem& find_problem(const Params& P, int tile) {
    int pi = 0;
#pragma unroll
    for (int i = 1; i < Params::kOps; ++i)
        if (i < P.head.n_problems && P.prob[i].tile_start <= tile) pi = i;
    return P.prob[pi];
}

// Column sums that the launch takes along: the epilogue warps have nothing to do until the first tile's main loop is over
// (0.3 us per 64-deep k-block), and a matrix of 8192 x 1024 is 14 KB per warp of the chip.  A warp takes a unit of kSumRows
// rows x 64 columns: 8 lanes cover a row's 128 bytes, eight loads of four rows in flight; the four rows of an instruction are
// added as a shuffle tree, so a unit's sum does not depend on which warp takes it.
// As a launch of its own between the products and the finishing launch this cost 9-15 us of every
// backward call on 8192 tokens, 1024 wide, sums and finishing launch together; now 4-5.
__device__ __forceinline__ void side_sums(const SideSums& S, int first, int stride, int lane) {
    int tiles = 0;
    for (int j = 0; j < S.n_jobs; ++j) tiles += S.col_tiles[j];
    for (int unit = first; unit < tiles * S.chunks; unit += stride) {
        int j = 0, ct = unit % tiles;
        const int chunk = unit / tiles;
        while (ct >= S.col_tiles[j]) ct -= S.col_tiles[j++];
        const int cols = S.cols[j], c0 = ct * 64 + (lane & 7) * 8;
        const int64_t ld = S.ld[j], r0 = static_cast<int64_t>(chunk) * kSumRows;
        const int nr = static_cast<int>(min(static_cast<int64_t>(kSumRows), S.rows - r0));
        const uint16_t* p = S.M[j] + r0 * ld + c0;
        float acc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = 0.f;
        if (S.vec_ok[j] && c0 + 8 <= cols) {
#pragma unroll 1
            for (int r = lane >> 3; r < nr; r += 32) {
                uint4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    v[u] = r + 4 * u < nr ? *reinterpret_cast<const uint4*>(p + (r + 4 * u) * ld) : make_uint4(0, 0, 0, 0);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    acc[0] += bf16_lo(v[u].x); acc[1] += bf16_hi(v[u].x);
                    acc[2] += bf16_lo(v[u].y); acc[3] += bf16_hi(v[u].y);
                    acc[4] += bf16_lo(v[u].z); acc[5] += bf16_hi(v[u].z);
                    acc[6] += bf16_lo(v[u].w); acc[7] += bf16_hi(v[u].w);
                }
            }
        } else {
#pragma unroll 1
            for (int r = lane >> 3; r < nr; r += 4)
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (c0 + e < cols) acc[e] += __uint_as_float(static_cast<uint32_t>(p[r * ld + e]) << 16);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 8);
            acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 16);
        }
        float* out = S.partial[j] + static_cast<int64_t>(chunk) * cols;
        if (lane < 8) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (c0 + e < cols) out[c0 + e] = acc[e];
        }
    }
}

// The sums of matrices of few rows, whole: the epilogue warps of a CTA take 64 columns together, warp w the rows 32 w .. 32 w + 31
// of every 256, and the eight sums of a column are added in order through shared memory (scratch: 2 KB), so that no finishing
// launch is needed.  (The step of a 320-token block with biases: 15 launches, 119 us; so 12, see kSumWholeRows.)
__device__ __forceinline__ void side_sums_whole(const SideSums& S, uint32_t scratch, int ew, int lane) {
    int tiles = 0;
    for (int j = 0; j < S.n_jobs; ++j) tiles += S.col_tiles[j];
    for (int unit = blockIdx.x; unit < tiles; unit += gridDim.x) {
        int j = 0, ct = unit;
        while (ct >= S.col_tiles[j]) ct -= S.col_tiles[j++];
        const int cols = S.cols[j], c0 = ct * 64 + (lane & 7) * 8, rows = static_cast<int>(S.rows);
        const int64_t ld = S.ld[j];
        const uint16_t* p = S.M[j] + c0;
        const bool vec = S.vec_ok[j] && c0 + 8 <= cols;
        float acc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = 0.f;
#pragma unroll 1
        for (int r0 = 32 * ew; r0 < rows; r0 += 32 * kEpiWarps) {
            const int r = r0 + (lane >> 3);
            if (vec) {
                uint4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = r + 4 * u < rows ? *reinterpret_cast<const uint4*>(p + (r + 4 * u) * ld) : make_uint4(0, 0, 0, 0);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    acc[0] += bf16_lo(v[u].x); acc[1] += bf16_hi(v[u].x);
                    acc[2] += bf16_lo(v[u].y); acc[3] += bf16_hi(v[u].y);
                    acc[4] += bf16_lo(v[u].z); acc[5] += bf16_hi(v[u].z);
                    acc[6] += bf16_lo(v[u].w); acc[7] += bf16_hi(v[u].w);
                }
            } else {
#pragma unroll 1
                for (int u = 0; u < 8; ++u)
                    if (r + 4 * u < rows)
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            if (c0 + e < cols) acc[e] += __uint_as_float(static_cast<uint32_t>(p[(r + 4 * u) * ld + e]) << 16);
            }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 8);
            acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 16);
        }
        if (lane < 8) {
#pragma unroll
            for (int e = 0; e < 8; ++e) asm volatile("st.shared.f32 [%0], %1;" ::"r"(scratch + 4 * (64 * ew + 8 * lane + e)), "f"(acc[e]) : "memory");
        }
        asm volatile("barrier.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");
        const int c = ct * 64 + 32 * ew + lane;
        if (ew < 2 && c < cols) {
            float t = 0.f;
#pragma unroll
            for (int w = 0; w < kEpiWarps; ++w) {
                float v;
                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(scratch + 4 * (64 * w + 32 * ew + lane)) : "memory");
                t += v;
            }
            if (S.out_f32) static_cast<float*>(S.out[j])[c] = t;
            else static_cast<__nv_bfloat16*>(S.out[j])[c] = __float2bfloat16_rn(t);
        }
        asm volatile("barrier.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");
    }
}

// ------------------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------------------
template <int FORM, typename Params>
__global__ void __launch_bounds__(kThreads, 1) gemm_kernel(const __grid_constant__ Params P) {
    constexpr bool PAIR = FORM == TILE_PAIR;
    constexpr int kTileM = TileShape<FORM>::kM, kTileN = TileShape<FORM>::kN;
    constexpr int kTmemCols = TileShape<FORM>::kTmemCols, kStages = TileShape<FORM>::kStages, kBStage = TileShape<FORM>::kBStage;
    constexpr int kHalfN = FORM == TILE_SLIM ? 64 : kTileN / 2;   // columns of an epilogue warp (64-wide tiles: of the first four)
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;       // 1024-byte aligned stage memory
    uint8_t* smem = smem_raw + (base - raw_addr);
    const uint32_t sA = base, sB = base + kStages * kSub * kAStage;
    const uint32_t sEpi = base + kRingBytes;
    uint8_t* tail = smem + kRingBytes + kEpiBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(tail);        // full[S], empty[S], tmem_full[2], tmem_empty[2]
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(tail + (2 * kMaxStages + 4) * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + (2 * kMaxStages + 4) * 8 + 8);
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
    auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * kStages + a); };
    auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * kStages + 2 + a); };

    // Launched with programmatic stream serialization: the next launch of this engine may place its CTAs as
    // soon as SMs free up and set itself up; it reads or writes no global memory before the wait below.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t cta_rank = PAIR ? cluster_ctarank() : 0u;   // 0 = leader: issues the MMAs, owns full/tmem_empty
    const bool leader = cta_rank == 0;
    const int worker = PAIR ? blockIdx.x >> 1 : blockIdx.x;
    const int n_workers = PAIR ? gridDim.x >> 1 : gridDim.x;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full_bar(s), 1);                // the leader's producer announces the bytes of both CTAs
            mbar_init(empty_bar(s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(tfull_bar(a), 1);
            mbar_init(tempty_bar(a), PAIR ? 2 * kEpiWarps : FORM == TILE_SLIM ? kEpiWarps / 2 : kEpiWarps);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const int tile0 = P.head.rounds > 0 ? scheduled_tile(P, worker, n_workers, 0) : -1;
        if (tile0 >= 0) {
            // warm the descriptors of the first tile while TMEM is allocated and the CTAs meet
            const DevProblem& Q0 = find_problem(P, tile0);
            prefetch_tensormap(&P.maps[Q0.map_a[0]]);
            prefetch_tensormap(&P.maps[Q0.map_b[0][cta_rank]]);
        }
    }
    if (warp == 1) {
        if (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync_all();     // the peer's barriers are initialised before anything signals them
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    // everything earlier in the stream has completed and its writes are visible after this
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------------ producer (both CTAs of a pair)
        if (elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int round = 0; ok && round < P.head.rounds; ++round) {
                const int tile = scheduled_tile(P, worker, n_workers, round);
                if (tile < 0) continue;
                const DevProblem& Q = find_problem(P, tile);
                const int local = tile - Q.tile_start;
                const int m0 = (local % Q.tiles_m) * kTileM + static_cast<int>(cta_rank) * BM;
                const int n0 = (local / Q.tiles_m) * Q.n_per_tile;
                // a stage carries up to kSub k-blocks of one K segment
                for (int seg = 0; ok && seg < kMaxSeg; ++seg) {
                const int kb_lo = seg ? Q.kb_end[seg - 1] : 0, kb_hi = Q.kb_end[seg];
                for (int kb0 = kb_lo; kb0 < kb_hi; kb0 += kSub) {
                    const int nsub = min(kSub, kb_hi - kb0);
                    if (!(ok = mbar_wait<PAIR>(empty_bar(stage), phase ^ 1u, abort_flag, 1, P.head.status, P.head.wait_limit_ns))) break;
                    // "big" operands arrive as one box holding both k-blocks (zero-filled past the end of K)
                    const bool a_big = PAIR && Q.a_big[seg], b_big = PAIR && Q.b_big[seg];
                    const uint32_t tx = (a_big ? kSub : nsub) * kAStage + (b_big ? kSub : nsub) * kBStage;
                    if (PAIR) {
                        if (leader) mbar_expect_tx(full_bar(stage), 2 * tx);   // both CTAs' bytes
                    } else {
                        mbar_expect_tx(full_bar(stage), tx);
                    }
                    if (PAIR && (a_big || b_big)) {
                        const int k0 = (kb0 - kb_lo) * BK + Q.k_off[seg];
                        const uint32_t fb = map_to_cta(full_bar(stage), 0);
                        if (a_big) {
                            const uint32_t dst = sA + stage * kSub * kAStage;
                            const CUtensorMap* ma = &P.maps[Q.map_a[seg]];
                            if (!Q.a_mn[seg]) {           // (64 k, 128 rows, 2 k-blocks)
                                if (leader) tma_load_3d(dst, ma, 0, m0, k0 >> 6, full_bar(stage));
                                else tma_load_3d_pair(dst, ma, 0, m0, k0 >> 6, fb);
                            } else {                      // (64 m, 64 k, 2 atoms, 2 k-blocks)
                                if (leader) tma_load_4d(dst, ma, 0, m0 >> 6, k0 >> 6, full_bar(stage));
                                else tma_load_4d_pair(dst, ma, 0, m0 >> 6, k0 >> 6, fb);
                            }
                        }
                        if (b_big) {
                            const uint32_t dst = sB + stage * kSub * kBStage;
                            const CUtensorMap* mb = &P.maps[Q.map_b[seg][cta_rank]];
                            const int nc = n0 + static_cast<int>(cta_rank) * Q.half1_n_off;
                            if (!Q.b_mn[seg]) {
                                if (leader) tma_load_3d(dst, mb, 0, nc, k0 >> 6, full_bar(stage));
                                else tma_load_3d_pair(dst, mb, 0, nc, k0 >> 6, fb);
                            } else {
                                if (leader) tma_load_4d(dst, mb, 0, nc >> 6, k0 >> 6, full_bar(stage));
                                else tma_load_4d_pair(dst, mb, 0, nc >> 6, k0 >> 6, fb);
                            }
                        }
                    }
#pragma unroll
                    for (int sub = 0; sub < kSub; ++sub) {
                    if (sub >= nsub) break;
                    const int kb = kb0 + sub;
                    const int k0 = (kb - kb_lo) * BK + Q.k_off[seg];
                    const uint32_t a_dst = sA + (stage * kSub + sub) * kAStage, b_dst = sB + (stage * kSub + sub) * kBStage;
                    const CUtensorMap* ma = &P.maps[Q.map_a[seg]];
                    if (PAIR) {
                        // This CTA's share of the stage, completed on the leader's barrier: the leader uses the
                        // plain form on its own barrier (measurably cheaper), the peer the pair form that may
                        // signal the other CTA's barrier.
                        const uint32_t fb = map_to_cta(full_bar(stage), 0);
                        auto load = [&](uint32_t dst, const CUtensorMap* map, int x, int y) {
                            if (leader) tma_load_2d(dst, map, x, y, full_bar(stage));
                            else tma_load_2d_pair(dst, map, x, y, fb);
                        };
                        auto load3 = [&](uint32_t dst, const CUtensorMap* map, int y, int z) {
                            if (leader) tma_load_3d(dst, map, 0, y, z, full_bar(stage));
                            else tma_load_3d_pair(dst, map, 0, y, z, fb);
                        };
                        if (a_big) {
                        } else if (!Q.a_mn[seg]) {
                            load(a_dst, ma, k0, m0);
                        } else if (Q.a_3d[seg]) {
                            load3(a_dst, ma, k0, m0 >> 6);
                        } else {
                            load(a_dst, ma, m0, k0);
                            load(a_dst + kAtomBytes, ma, m0 + 64, k0);
                        }
                        const CUtensorMap* mb = &P.maps[Q.map_b[seg][cta_rank]];
                        const int nc = n0 + static_cast<int>(cta_rank) * Q.half1_n_off;
                        if (b_big) {
                        } else if (!Q.b_mn[seg]) {
                            load(b_dst, mb, k0, nc);
                        } else if (Q.b_3d[seg]) {
                            load3(b_dst, mb, k0, nc >> 6);
                        } else {
                            load(b_dst, mb, nc, k0);
                            load(b_dst + kAtomBytes, mb, nc + 64, k0);
                        }
                    } else {
                        if (!Q.a_mn[seg]) {
                            tma_load_2d(a_dst, ma, k0, m0, full_bar(stage));                    // box 64(k) x 128(m)
                        } else if (Q.a_3d[seg]) {
                            tma_load_3d(a_dst, ma, 0, k0, m0 >> 6, full_bar(stage));            // box 64 x 64(k) x 2 atoms
                        } else {
                            tma_load_2d(a_dst, ma, m0, k0, full_bar(stage));                    // box 64(m) x 64(k)
                            tma_load_2d(a_dst + kAtomBytes, ma, m0 + 64, k0, full_bar(stage));
                        }
#pragma unroll
                        for (int h = 0; h < (FORM == TILE_SLIM ? 1 : 2); ++h) {                 // half of the tile's columns of B each (64-wide tiles: all)
                            const CUtensorMap* mb = &P.maps[Q.map_b[seg][h]];
                            const int nc = n0 + h * Q.half1_n_off;
                            const uint32_t dst = b_dst + h * (kBStage / 2);
                            if (!Q.b_mn[seg]) {
                                tma_load_2d(dst, mb, k0, nc, full_bar(stage));                  // box 64(k) x kHalfN(n)
                            } else if (FORM == TILE_WIDE && Q.b_3d[seg]) {
                                tma_load_3d(dst, mb, 0, k0, nc >> 6, full_bar(stage));          // box 64 x 64(k) x 2 atoms
                            } else {
                                tma_load_2d(dst, mb, nc, k0, full_bar(stage));                  // box 64(n) x 64(k)
                                if (FORM == TILE_WIDE) tma_load_2d(dst + kAtomBytes, mb, nc + 64, k0, full_bar(stage));
                            }
                        }
                    }
                    }   // sub
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }   // kb0
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leader CTA only)
        if (leader && elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            int it = 0;
            bool ok = true;
            for (int round = 0; ok && round < P.head.rounds; ++round) {
                const int tile = scheduled_tile(P, worker, n_workers, round);
                if (tile < 0) continue;
                const DevProblem& Q = find_problem(P, tile);
                const int acc = it & 1;
                const uint32_t acc_phase = (it >> 1) & 1u;
                if (!(ok = mbar_wait<PAIR>(tempty_bar(acc), acc_phase ^ 1u, abort_flag, 2, P.head.status, P.head.wait_limit_ns))) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * kTileN;
                for (int seg = 0; ok && seg < kMaxSeg; ++seg) {
                const int kb_lo = seg ? Q.kb_end[seg - 1] : 0, kb_hi = Q.kb_end[seg];
                for (int kb0 = kb_lo; kb0 < kb_hi; kb0 += kSub) {
                    const int nsub = min(kSub, kb_hi - kb0);
                    if (!(ok = mbar_wait<PAIR>(full_bar(stage), phase, abort_flag, 3, P.head.status, P.head.wait_limit_ns))) break;
                    tc_fence_after();
#pragma unroll
                    for (int sub = 0; sub < kSub; ++sub) {
                        if (sub >= nsub) break;
                        const int kb = kb0 + sub;
                        const uint32_t a_mn = Q.a_mn[seg], b_mn = Q.b_mn[seg];
                        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (a_mn << 15) | (b_mn << 16) |
                                               (static_cast<uint32_t>(kTileN >> 3) << 17) | (static_cast<uint32_t>(kTileM >> 4) << 24);
                        const uint64_t a_desc = make_smem_desc(sA + (stage * kSub + sub) * kAStage, a_mn ? kAtomBytes : 16, 1024);
                        const uint64_t b_desc = make_smem_desc(sB + (stage * kSub + sub) * kBStage, b_mn ? kAtomBytes : 16, 1024);
                        const uint64_t a_step = a_mn ? (2048 >> 4) : (32 >> 4);   // per 16 k: two 8-row groups, or 32 bytes
                        const uint64_t b_step = b_mn ? (2048 >> 4) : (32 >> 4);
#pragma unroll
                        for (int ks = 0; ks < BK / 16; ++ks) {
                            if (PAIR) tc_mma_bf16_pair(d_tmem, a_desc + ks * a_step, b_desc + ks * b_step, idesc, (kb | ks) != 0 ? 1u : 0u);
                            else tc_mma_bf16(d_tmem, a_desc + ks * a_step, b_desc + ks * b_step, idesc, (kb | ks) != 0 ? 1u : 0u);
                        }
                    }
                    // the stage is free (in both CTAs) once these MMAs have read it
                    if (PAIR) {
                        tc_commit_pair(map_to_cta(empty_bar(stage), 0));
                        tc_commit_pair(map_to_cta(empty_bar(stage), 1));
                    } else {
                        tc_commit(empty_bar(stage));
                    }
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }
                }   // seg
                if (ok) {                              // accumulator complete (in both CTAs)
                    if (PAIR) {
                        tc_commit_pair(map_to_cta(tfull_bar(acc), 0));
                        tc_commit_pair(map_to_cta(tfull_bar(acc), 1));
                    } else {
                        tc_commit(tfull_bar(acc));
                    }
                }
                ++it;
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int ew = warp - 2;
        const int quad = warp & 3;            // TMEM lanes this warp may read: [32*quad, 32*quad + 32)
        const int half = ew >> 2;             // which half of the tile's columns
        const uint32_t buf_out = sEpi + ew * 2 * kEpiSlotBytes, buf_in = buf_out + kEpiSlotBytes;
        if (P.head.side.whole) side_sums_whole(P.head.side, sEpi, ew, lane);
        else if (P.head.side.n_jobs > 0) side_sums(P.head.side, blockIdx.x + gridDim.x * ew, gridDim.x * kEpiWarps, lane);
        int it = 0;
        bool ok = true;
        const int rounds = FORM == TILE_SLIM && half == 1 ? 0 : P.head.rounds;
        for (int round = 0; ok && round < rounds; ++round) {
            const int tile = scheduled_tile(P, worker, n_workers, round);
            if (tile < 0) continue;
            const DevProblem& Q = find_problem(P, tile);
            const int local = tile - Q.tile_start;
            const int m_warp = (local % Q.tiles_m) * kTileM + static_cast<int>(cta_rank) * BM + quad * 32;   // first row of this warp
            const int n0 = (local / Q.tiles_m) * Q.n_per_tile;
            const int acc = it & 1;
            const uint32_t acc_phase = (it >> 1) & 1u;
            const int epi = Q.epi;
            const int QM = Q.M, QN = Q.N;
            const CUtensorMap* mc0 = &P.maps[Q.map_c[0]];
            const CUtensorMap* mc1 = &P.maps[Q.map_c[1]];
            const CUtensorMap* mc2 = &P.maps[Q.map_c[2]];
            // saved activations of the derivative epilogues: first chunk requested before the accumulator is ready
            const bool need_h = epi >= EPI_DGELU_ERF;
            const bool need_hb = epi == EPI_DSWIGLU;
            const unsigned short* Hp = static_cast<const unsigned short*>(Q.H);
            const unsigned short* Hbp = static_cast<const unsigned short*>(Q.Hb);
            uint4 hq[4], hbq[4];
            if (need_h) staged_load32_issue(Hp, Q.ldh, m_warp, n0 + half * kHalfN, QM, QN, hq, lane);
            if (need_hb) staged_load32_issue(Hbp, Q.ldh, m_warp, n0 + half * kHalfN, QM, QN, hbq, lane);
            // the second slot doubles as the landing buffer of those loads: no store of an earlier tile may still read it
            if (need_h) stage_begin<0>(lane);
            // bias of this warp's columns, one column per lane and 32-column chunk (fetched while the tile is computed)
            float breg[4] = {0.f, 0.f, 0.f, 0.f};
            const bool has_bias = Q.bias != nullptr;
            if (has_bias) {
#pragma unroll
                for (int j = 0; j < kHalfN / 32; ++j) {
                    const int col = n0 + half * kHalfN + 32 * j + lane;
                    if (col < QN)
                        breg[j] = Q.bias_f32 ? static_cast<const float*>(Q.bias)[col]
                                             : __uint_as_float(static_cast<uint32_t>(static_cast<const unsigned short*>(Q.bias)[col]) << 16);
                }
            }
            if (!(ok = mbar_wait<PAIR>(tfull_bar(acc), acc_phase, abort_flag, 4, P.head.status, P.head.wait_limit_ns))) break;
            tc_fence_after();
            const uint32_t t_row = tmem_base + acc * kTileN + (static_cast<uint32_t>(quad * 32) << 16);
            const bool warp_rows = m_warp < QM;          // any row of this warp inside the output
            if (epi == EPI_SWIGLU) {
                // accumulator columns: gate, then up, for hidden units n0 .. n0 + kHalfN - 1.
                // The three outputs of a chunk alternate between the two slots, one store may stay in flight.
                int slot = 0;
                bool fresh = true;
                auto put = [&](const CUtensorMap* map, int n, const float (&v)[32]) {
                    if (fresh) stage_begin<0>(lane); else stage_begin<1>(lane);
                    fresh = false;
                    const uint32_t sb = buf_out + slot * kEpiSlotBytes;
                    stage_bf16x32(sb, lane, v);
                    stage_commit(map, sb, n, m_warp, lane);
                    slot ^= 1;
                };
#pragma unroll 1
                for (int c = 0; c < kHalfN / 64; ++c) {
                    const int hc = half * (kHalfN / 2) + c * 32;
                    uint32_t rg[32], ru[32];
                    tc_ld32(t_row + hc, rg);
                    tc_ld32(t_row + kHalfN + hc, ru);
                    tc_wait_ld();
                    const int n = n0 + hc;
                    if (n >= QN || !warp_rows) continue;
                    float g[32], u[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        g[i] = __uint_as_float(rg[i]);
                        u[i] = __uint_as_float(ru[i]);
                    }
                    put(mc0, n, g);
                    put(mc1, n, u);
#pragma unroll
                    for (int i = 0; i < 32; ++i) g[i] = g[i] * sigmoidf_(g[i]) * u[i];
                    put(mc2, n, g);
                }
            } else if (epi == EPI_STORE && !Q.out_f32) {
                // bf16 output: chunks of 64 columns, each one 32 x 128-byte image
#pragma unroll 1
                for (int c = 0; c < kHalfN / 64; ++c) {
                    const int col = half * kHalfN + c * 64;
                    uint32_t r0[32], r1[32];
                    tc_ld32(t_row + col, r0);
                    tc_ld32(t_row + col + 32, r1);
                    tc_wait_ld();
                    const int n = n0 + col;
                    if (n >= QN || !warp_rows) continue;
                    float v0[32], v1[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        v0[i] = __uint_as_float(r0[i]);
                        v1[i] = __uint_as_float(r1[i]);
                    }
                    if (has_bias) {
                        add_bias32(v0, c ? breg[2] : breg[0]);
                        add_bias32(v1, c ? breg[3] : breg[1]);
                    }
                    stage_begin<0>(lane);
                    stage_bf16x64(buf_out, lane, v0, v1);
                    stage_commit(mc0, buf_out, n, m_warp, lane, Q.accumulate != 0);
                }
            } else if (epi == EPI_GELU_ERF || epi == EPI_GELU_TANH) {
                // H = acc + bias and A = GELU(H), 64 columns at a time
#pragma unroll 1
                for (int c = 0; c < kHalfN / 64; ++c) {
                    const int col = half * kHalfN + c * 64;
                    uint32_t r0[32], r1[32];
                    tc_ld32(t_row + col, r0);
                    tc_ld32(t_row + col + 32, r1);
                    tc_wait_ld();
                    const int n = n0 + col;
                    if (n >= QN || !warp_rows) continue;
                    float v0[32], v1[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        v0[i] = __uint_as_float(r0[i]);
                        v1[i] = __uint_as_float(r1[i]);
                    }
                    if (has_bias) {
                        add_bias32(v0, c ? breg[2] : breg[0]);
                        add_bias32(v1, c ? breg[3] : breg[1]);
                    }
                    stage_begin<0>(lane);
                    stage_bf16x64(buf_out, lane, v0, v1);
                    stage_commit(mc0, buf_out, n, m_warp, lane);
                    if (epi == EPI_GELU_ERF) {
                        gelu_erf32(v0);
                        gelu_erf32(v1);
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            v0[i] = gelu_tanh(v0[i]);
                            v1[i] = gelu_tanh(v1[i]);
                        }
                    }
                    stage_begin<0>(lane);
                    stage_bf16x64(buf_out, lane, v0, v1);
                    stage_commit(mc1, buf_out, n, m_warp, lane);
                }
            } else {
                // 32 columns at a time: fp32 outputs and the derivative epilogues
#pragma unroll 1
                for (int c = 0; c < kHalfN / 32; ++c) {
                    const int col = half * kHalfN + c * 32;
                    uint32_t r[32];
                    tc_ld32(t_row + col, r);
                    tc_wait_ld();
                    const int n = n0 + col;
                    const int nv = min(32, QN - n);
                    if (nv <= 0) continue;
                    float v[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
                    if (has_bias) add_bias32(v, c == 0 ? breg[0] : c == 1 ? breg[1] : c == 2 ? breg[2] : breg[3]);
                    if (epi == EPI_STORE) {                // fp32 output: one 32 x 128-byte image
                        if (warp_rows) {
                            stage_begin<0>(lane);
                            stage_f32x32(buf_out, lane, v);
                            stage_commit(mc0, buf_out, n, m_warp, lane, Q.accumulate != 0);
                        }
                    } else if (epi == EPI_DGELU_ERF || epi == EPI_DGELU_TANH) {
                        float h[32];
                        staged_load32_finish(buf_in, hq, h, lane);
                        if (c + 1 < kHalfN / 32) staged_load32_issue(Hp, Q.ldh, m_warp, n + 32, QM, QN, hq, lane);
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (epi != EPI_DGELU_ERF) v[i] *= dgelu_tanh(h[i]);
                        if (epi == EPI_DGELU_ERF) dgelu_erf32(v, h);
                        if (warp_rows) {
                            stage_begin<0>(lane);
                            stage_bf16x32(buf_out, lane, v);
                            stage_commit(mc0, buf_out, n, m_warp, lane);
                        }
                    } else {  // EPI_DSWIGLU
                        float hg[32], hu[32];
                        staged_load32_finish(buf_in, hq, hg, lane);
                        staged_load32_finish(buf_in, hbq, hu, lane);
                        if (c + 1 < kHalfN / 32) {
                            staged_load32_issue(Hp, Q.ldh, m_warp, n + 32, QM, QN, hq, lane);
                            staged_load32_issue(Hbp, Q.ldh, m_warp, n + 32, QM, QN, hbq, lane);
                        }
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            const float s = sigmoidf_(hg[i]);
                            hu[i] = v[i] * hu[i] * s * (1.f + hg[i] * (1.f - s));   // dH_gate
                            v[i] = v[i] * hg[i] * s;                                // dH_up
                        }
                        if (warp_rows) {
                            stage_begin<0>(lane);
                            stage_bf16x32(buf_out, lane, hu);
                            stage_commit(mc0, buf_out, n, m_warp, lane);
                            stage_begin<0>(lane);
                            stage_bf16x32(buf_out, lane, v);
                            stage_commit(mc1, buf_out, n, m_warp, lane);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {                       // the accumulator may be overwritten: tell the MMA issuer
                if (PAIR) mbar_arrive_cluster(map_to_cta(tempty_bar(acc), 0));
                else mbar_arrive(tempty_bar(acc));
            }
            ++it;
        }
        bulk_wait_all();                           // this warp's tile stores have landed
    }

    // ---------------------------------------------------------------------- teardown
    __syncwarp();
    if (*abort_flag) {
        // give copies that are still in flight time to land before the shared memory is released
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync_all();     // neither CTA leaves while the other may still signal its barriers
    if (warp == 1) {
        tc_fence_after();
        if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                              const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn get_encode() {
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

// MN-major operand whose row length is a multiple of 64: the matrix [K][MN] viewed as (64, K, MN/64) with strides
// (2 B, pitch, 128 B), so that one box of 64 x 64 x 2 brings both 64-wide swizzle atoms of a 128-wide slab
// in the atom-major order the MMA descriptor expects.  Returns false when the view cannot be encoded.
bool encode_map_mn3d(CUtensorMap* out, const Stored& s) {
    EncodeFn enc = get_encode();
    if (!enc || !s.ptr || s.cols % 64 != 0 || !aligned16(s.ptr) || (s.ld * 2) % 16 != 0) return false;
    const cuuint64_t dims[3] = {64, static_cast<cuuint64_t>(s.rows), static_cast<cuuint64_t>(s.cols / 64)};
    const cuuint64_t strides[2] = {static_cast<cuuint64_t>(s.ld) * 2, 128};
    const cuuint32_t box[3] = {64, 64, 2};
    const cuuint32_t estr[3] = {1, 1, 1};
    return enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(s.ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Pair mode, one box per operand per stage (two 64-deep k-blocks), when the extents are multiples of 64:
//   K-major  [rows][K]  viewed as (64, rows, K/64)          box 64 x 128 x 2        -> [k-block][row][64 k]
//   MN-major [K][MN]    viewed as (64, 64, MN/64, K/64)     box 64 x 64 x 2 x 2     -> [k-block][atom][k][64 mn]
// Both orders are exactly two consecutive k-block images of the per-k-block layout.
bool encode_map_big(CUtensorMap* out, const Stored& s, bool mn) {
    EncodeFn enc = get_encode();
    if (!enc || !s.ptr || s.cols % 64 != 0 || !aligned16(s.ptr) || (s.ld * 2) % 16 != 0) return false;
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    if (!mn) {
        const cuuint64_t dims[3] = {64, static_cast<cuuint64_t>(s.rows), static_cast<cuuint64_t>(s.cols / 64)};
        const cuuint64_t strides[2] = {static_cast<cuuint64_t>(s.ld) * 2, 128};
        const cuuint32_t box[3] = {64, 128, 2};
        return enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(s.ptr), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    if (s.rows % 64 != 0) return false;
    const cuuint64_t dims[4] = {64, 64, static_cast<cuuint64_t>(s.cols / 64), static_cast<cuuint64_t>(s.rows / 64)};
    const cuuint64_t strides[3] = {static_cast<cuuint64_t>(s.ld) * 2, 128, static_cast<cuuint64_t>(s.ld) * 128};
    const cuuint32_t box[4] = {64, 64, 2, 2};
    return enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(s.ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tensor map of a stored row-major bf16 matrix; box = 64 elements along the row x box_rows rows
// (128-byte swizzle, operand loads), or 32 x 32 with the 64-byte swizzle (epilogue stores).
ecospa_status_t encode_map(CUtensorMap* out, const Stored& s, int box_rows, bool store_box = false) {
    EncodeFn enc = get_encode();
    if (!enc) {
        set_cuda_error(cudaErrorNotSupported, "cuTensorMapEncodeTiled entry point");
        return ECOSPA_ERR_CUDA;
    }
    if (!s.ptr || s.rows < 1 || s.cols < 1 || s.ld < s.cols) return ECOSPA_ERR_INVALID;
    if (!aligned16(s.ptr) || (s.ld * 2) % 16 != 0) return ECOSPA_ERR_ALIGNMENT;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(s.cols), static_cast<cuuint64_t>(s.rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(s.ld) * 2};
    const cuuint32_t box[2] = {store_box ? 32u : 64u, static_cast<cuuint32_t>(box_rows)};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(s.ptr), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, store_box ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
        return ECOSPA_ERR_CUDA;
    }
    return ECOSPA_OK;
}

// Store map of an output (rows x cols, pitch ld elements): boxes of 32 rows x 64 bf16 or 32 fp32 columns
// (128-byte swizzle) or 32 rows x 32 bf16 columns (64-byte swizzle), matching the staging images.
ecospa_status_t encode_out_map(CUtensorMap* out, void* ptr, int64_t rows, int64_t cols, int64_t ld, bool f32, bool wide) {
    EncodeFn enc = get_encode();
    if (!enc) {
        set_cuda_error(cudaErrorNotSupported, "cuTensorMapEncodeTiled entry point");
        return ECOSPA_ERR_CUDA;
    }
    const int eb = f32 ? 4 : 2;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld) * eb};
    const cuuint32_t box[2] = {(f32 || !wide) ? 32u : 64u, 32u};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(out, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ptr, dims, strides, box,
                           estr, CU_TENSOR_MAP_INTERLEAVE_NONE, (f32 || wide) ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                           CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled (output)");
        return ECOSPA_ERR_CUDA;
    }
    return ECOSPA_OK;
}

// Per-device facts of the engine, looked up the first time a device is used (with that device current).
constexpr int kMaxDevices = 64;
struct DeviceState {
    std::once_flag once;
    ecospa_status_t st = ECOSPA_OK;
    int num_sms = 0;
    int max_pairs = 0;      // CTA pairs that can be resident at once (clusters must fit inside a GPC)
    int* status_ptr = nullptr;   // this device's copy of g_gemm_status
};
DeviceState g_dev[kMaxDevices];
int g_pair_mode = 1;   // 0: no CTA pairs (cta_group::2); 1: as launch_grouped_gemm decides
std::atomic<unsigned long long> g_wait_limit_ns{kDefaultWaitLimitNs};

template <typename Params>
cudaError_t allow_smem(void (*kernel)(Params)) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes); }

// State of the current device (set up on first use), or nullptr with *st set.
DeviceState* gemm_setup(ecospa_status_t* st_out) {
    int dev = 0;
    cudaError_t e0 = cudaGetDevice(&dev);
    if (e0 != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        if (e0 != cudaSuccess) {
            set_cuda_error(e0, "gemm setup (cudaGetDevice)");
            cudaGetLastError();
        }
        *st_out = e0 != cudaSuccess ? ECOSPA_ERR_CUDA : ECOSPA_ERR_UNSUPPORTED;
        return nullptr;
    }
    DeviceState& D = g_dev[dev];
    std::call_once(D.once, [&D, dev] {
        cudaError_t e = cudaDeviceGetAttribute(&D.num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = allow_smem(gemm_kernel<TILE_SINGLE, SmallParams>);
        if (e == cudaSuccess) e = allow_smem(gemm_kernel<TILE_SINGLE, LargeParams>);
        if (e == cudaSuccess) e = allow_smem(gemm_kernel<TILE_SLIM, SmallParams>);
        if (e == cudaSuccess) e = allow_smem(gemm_kernel<TILE_SLIM, LargeParams>);
        if (e == cudaSuccess) e = allow_smem(gemm_kernel<TILE_WIDE, SmallParams>);
        if (e == cudaSuccess) e = allow_smem(gemm_kernel<TILE_WIDE, LargeParams>);
        if (e == cudaSuccess) e = allow_smem(gemm_kernel<TILE_PAIR, SmallParams>);
        if (e == cudaSuccess) e = allow_smem(gemm_kernel<TILE_PAIR, LargeParams>);
        if (const char* v = std::getenv("ECOSPA_GEMM_PAIR")) g_pair_mode = std::atoi(v);
        if (e == cudaSuccess) {
            // the tile schedule is static, so only as many pairs as can run at the same time are launched
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(2 * (D.num_sms / 2));
            cfg.blockDim = dim3(kThreads);
            cfg.dynamicSmemBytes = kSmemBytes;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 2;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, gemm_kernel<TILE_PAIR, LargeParams>, &cfg) == cudaSuccess && n > 0) D.max_pairs = n;
            else cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaGetSymbolAddress(reinterpret_cast<void**>(&D.status_ptr), g_gemm_status);
        if (e != cudaSuccess) {
            set_cuda_error(e, "gemm setup");
            cudaGetLastError();
            D.st = ECOSPA_ERR_CUDA;
        }
    });
    *st_out = D.st;
    return D.st == ECOSPA_OK ? &D : nullptr;
}

// Tile schedule.  Tiles are numbered op by op, longest contraction first.  With few tiles per worker the
// plain stride (worker w takes w, w + workers, ...) can leave one worker with several long tiles, so the
// tiles are handed out longest first to the least-loaded worker (ties: lowest worker) and the result is
// written as a table; with many tiles per worker the stride is balanced enough and needs no table.
void build_schedule(LargeParams& gp, int workers) {
    const int tiles = gp.head.total_tiles;
    gp.head.use_order = 0;
    gp.head.rounds = static_cast<int32_t>(ceil_div(tiles, workers));
    if (tiles <= workers || tiles > LargeParams::kOrder || tiles >= kNoTile) return;
    // workers as a binary heap by (load, worker): the top is the least loaded one, the lowest of those with equal loads
    static thread_local uint64_t heap[256];
    static thread_local int32_t len[256];
    static thread_local uint16_t lists[256][64];
    if (workers > 256) return;
    for (int w = 0; w < workers; ++w) {
        heap[w] = static_cast<uint64_t>(w);
        len[w] = 0;
    }
    int max_len = 0;
    int pi = 0;
    for (int t = 0; t < tiles; ++t) {
        while (pi + 1 < gp.head.n_problems && gp.prob[pi + 1].tile_start <= t) ++pi;
        // main loop, or the epilogue where that is the longer of the two (measured, in k-block times), + a fixed share
        static const int kEpiCost[7] = {5, 14, 14, 16, 20, 20, 26};
        const int64_t cost = std::max<int64_t>(gp.prob[pi].kblocks, kEpiCost[gp.prob[pi].epi]) + 4;
        const int best = static_cast<int>(heap[0] & 0xff);
        if (len[best] >= 64) return;                       // not expected; keep the stride
        lists[best][len[best]++] = static_cast<uint16_t>(t);
        max_len = std::max(max_len, static_cast<int>(len[best]));
        const uint64_t key = heap[0] + (static_cast<uint64_t>(cost) << 8);
        int i = 0;                                         // sift the new load down
        for (int c = 1; c < workers; c = 2 * i + 1) {
            if (c + 1 < workers && heap[c + 1] < heap[c]) ++c;
            if (heap[c] >= key) break;
            heap[i] = heap[c];
            i = c;
        }
        heap[i] = key;
    }
    if (static_cast<int64_t>(max_len) * workers > LargeParams::kOrder) return;
    for (int i = 0; i < max_len; ++i)
        for (int w = 0; w < workers; ++w) gp.order[w + i * workers] = i < len[w] ? lists[w][i] : kNoTile;
    gp.head.rounds = max_len;
    gp.head.use_order = 1;
}

// The maps of a launch: operands that several products (or both halves of a tile) share get one map.
struct MapTable {
    struct Key {
        const void* ptr;
        int64_t rows, cols, ld;
        int form;
    };
    static constexpr int kOutput = 16;                     // (no operand form has this value)
    LargeParams& gp;
    Key key[LargeParams::kMaps];
    int n = 0;
    explicit MapTable(LargeParams& g) : gp(g) {}
    int find(const Stored& m, int form) const {
        for (int i = 0; i < n; ++i)
            if (key[i].ptr == m.ptr && key[i].rows == m.rows && key[i].cols == m.cols && key[i].ld == m.ld && key[i].form == form) return i;
        return -1;
    }
    CUtensorMap* next() { return n < LargeParams::kMaps ? &gp.maps[n] : nullptr; }
    int add(const Stored& m, int form) {
        key[n] = Key{m.ptr, m.rows, m.cols, m.ld, form};
        return n++;
    }
};
enum OperandForm { FORM_PLAIN = 0, FORM_3D = 1, FORM_BIG = 2 };   // how a stage's box is fetched, see the encoders
// Map of operand m (K-major or MN-major) in the widest form that it and the launch's mode allow; box_rows: of the plain
// K-major form.
ecospa_status_t operand_map(MapTable& T, const Stored& m, bool mn, bool pair, int box_rows, bool allow_3d, int* map, int* form) {
    // what tells the maps of one tensor apart: form, orientation and, for the plain K-major form, the box
    auto tag = [&](int f) { return 4 * f + (mn ? 2 : 0) + (f == FORM_PLAIN && !mn && box_rows != 128 ? 1 : 0); };
    for (int f = pair ? FORM_BIG : FORM_3D; f >= FORM_PLAIN; --f) {
        if (f == FORM_3D && !allow_3d) continue;
        const int id = T.find(m, tag(f));
        if (id >= 0) {
            *map = id;
            *form = f;
            return ECOSPA_OK;
        }
    }
    CUtensorMap* out = T.next();
    if (!out) return ECOSPA_ERR_UNSUPPORTED;               // (not reached by the library's own calls)
    if (pair && encode_map_big(out, m, mn)) *form = FORM_BIG;
    else if (allow_3d && mn && encode_map_mn3d(out, m)) *form = FORM_3D;
    else {
        const ecospa_status_t st = encode_map(out, m, mn ? 64 : box_rows);
        if (st != ECOSPA_OK) return st;
        *form = FORM_PLAIN;
    }
    *map = T.add(m, tag(*form));
    return ECOSPA_OK;
}

template <int FORM, typename Params>
cudaError_t launch_form(const Params& gp, int workers, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(FORM == TILE_PAIR ? 2 * workers : workers);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = FORM == TILE_PAIR ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, gemm_kernel<FORM, Params>, gp);
}
template <int FORM>
cudaError_t launch_smallest_form(const LargeParams& gp, int n_maps, int workers, cudaStream_t stream) {
    const int n_order = gp.head.use_order ? gp.head.rounds * workers : 0;
    if (n_maps > SmallParams::kMaps || gp.head.n_problems > SmallParams::kOps || n_order > SmallParams::kOrder)
        return launch_form<FORM>(gp, workers, stream);
    static thread_local SmallParams sp;
    std::memcpy(sp.maps, gp.maps, n_maps * sizeof(CUtensorMap));
    std::memcpy(sp.prob, gp.prob, gp.head.n_problems * sizeof(DevProblem));
    sp.head = gp.head;
    std::memcpy(sp.order, gp.order, n_order * sizeof(uint16_t));
    return launch_form<FORM>(sp, workers, stream);
}

}  // namespace

// Host-only checks of a launch (no CUDA call): shapes, pointers, 16-byte alignment of every base and pitch.
ecospa_status_t validate_gemm_ops(const GemmOp* ops, int n_ops) {
    if (!ops || n_ops < 1 || n_ops > kMaxGemmOps) return ECOSPA_ERR_INVALID;
    for (int i = 0; i < n_ops; ++i) {
        const GemmOp& op = ops[i];
        if (op.M < 1 || op.N < 1 || op.n_kseg < 1 || op.n_kseg > kMaxSeg || !op.C || op.ldc < 1) return ECOSPA_ERR_INVALID;
        if (op.M > INT32_MAX || op.N > INT32_MAX) return ECOSPA_ERR_INVALID;
        if (op.epi < EPI_STORE || op.epi > EPI_DSWIGLU) return ECOSPA_ERR_INVALID;
        const int out_eb = op.out_f32 ? 4 : 2;
        if (!aligned16(op.C) || (op.ldc * out_eb) % 16) return ECOSPA_ERR_ALIGNMENT;
        if (op.ldc < op.N) return ECOSPA_ERR_INVALID;
        if (op.bias && !aligned16(op.bias)) return ECOSPA_ERR_ALIGNMENT;
        for (int s = 0; s < op.n_kseg; ++s) {
            const KSegment& ks = op.seg[s];
            if (ks.K < 1 || ks.k_begin < 0 || ks.k_begin % BK) return ECOSPA_ERR_INVALID;
            const Stored* mats[3] = {&ks.a, &ks.b[0], op.epi == EPI_SWIGLU ? &ks.b[1] : nullptr};
            for (const Stored* m : mats) {
                if (!m) continue;
                if (!m->ptr || m->rows < 1 || m->cols < 1 || m->ld < m->cols) return ECOSPA_ERR_INVALID;
                if (!aligned16(m->ptr) || (m->ld * 2) % 16) return ECOSPA_ERR_ALIGNMENT;
            }
        }
    }
    return ECOSPA_OK;
}

ecospa_status_t launch_grouped_gemm(const GemmOp* ops, int n_ops, cudaStream_t stream, const SideSums* side) {
    ecospa_status_t st = validate_gemm_ops(ops, n_ops);
    if (st != ECOSPA_OK) return st;
    DeviceState* dev = gemm_setup(&st);
    if (!dev) return st;
    const int g_max_pairs = dev->max_pairs, g_num_sms = dev->num_sms;

    // longest contraction first
    int order[kMaxGemmOps];
    int64_t ktot[kMaxGemmOps];
    for (int i = 0; i < n_ops; ++i) {
        order[i] = i;
        ktot[i] = 0;
        for (int s = 0; s < ops[i].n_kseg; ++s) ktot[i] += ceil_div(ops[i].seg[s].K, BK);
    }
    std::stable_sort(order, order + n_ops, [&](int a, int b) { return ktot[a] > ktot[b]; });

    // CTA pairs fetch a third less operand data per flop, but their 256x256 tiles leave most of the chip idle in a small
    // product, and a lone launch then waits for one pair's main loop and for an epilogue of 128x256 outputs per CTA.  Where
    // 128x128 tiles of single CTAs still fit one round, they take their place (320 tokens, 768 wide: the eight products of a training step took 10-19 us each and take 8-16).
    // Beyond one round pairs need rows for both CTAs: launches of at most 128 rows (few tokens) take single CTAs with 128x256
    // tiles (Q/K/V of an 8192-wide model, 16 to 128 tokens: pairs 99-103 us, 128x128 tiles 86-89, 128x256 80-82; up to 4 tokens, where
    // every tile waits for the same few lines of X, 117, 120 and 123).
    // Where tiles of half that width fit one round too, they take it: an SM then fetches 24 KB instead of 32 per 64-deep k-block, twice
    // as many SMs fetch, and a tile's epilogue is half as long: 113 -> 103 us for the training step of 320 tokens, 768 wide.  (Not for
    // the gated epilogue, whose tile is two operands side by side.)
    // But not many of them on few rows: all tiles then wait for the same few lines of X, k-block by k-block, and twice as many wait
    // twice as long.  Measured, this holds while X takes less than 128 KB and there are more than 48 tiles, or with contractions
    // above 4096 more than 32.  128 x 64 / 128 x 128 tiles, us: Q/K/V of 4096 / 2048 (96 narrow tiles) 28.6 / 20.9 at 8 tokens, 13.9 / 15 at 16
    // (128 KB); of 2048 / 2048 17.9 / 11.6 at one, 14.8 / 10.3 at 24, 8.7 / 11 at 32; 1024 / 6144 (96) 9.6 / 7.0 at one, 6.1 / 7.5 at 64; 2048 /
    // 2560 (40) 10.3 / 10.6; 768 / 3072 (48) 5.5 / 6.4; 8192 / 2688 (42) 32.8 / 27.4 at one, 23.9 / 31.8 at 8.
    int64_t single_tiles = 0, slim_tiles = 0;
    bool any_tall = false;
    int64_t x_bytes = 0, k_max = 0;                            // X: operand A
    for (int i = 0; i < n_ops; ++i) {
        int64_t k = 0;
        for (int s = 0; s < ops[i].n_kseg; ++s) k += ops[i].seg[s].K;
        k_max = std::max(k_max, k);
        x_bytes = std::max(x_bytes, 2 * std::min<int64_t>(ops[i].M, BM) * k);
        const int per_tile = ops[i].epi == EPI_SWIGLU ? TileShape<TILE_SINGLE>::kN / 2 : TileShape<TILE_SINGLE>::kN;
        single_tiles += ceil_div(ops[i].M, BM) * ceil_div(ops[i].N, per_tile);
        slim_tiles += ops[i].epi == EPI_SWIGLU ? g_num_sms + 1 : ceil_div(ops[i].M, BM) * ceil_div(ops[i].N, TileShape<TILE_SLIM>::kN);
        any_tall = any_tall || ops[i].M > BM;
    }
    const bool pairs = g_pair_mode != 0 && g_max_pairs >= 1 && any_tall;
    const bool crowded = !any_tall && x_bytes < 128 * 1024 && slim_tiles > (k_max > 4096 ? 32 : 48);
    const int form = slim_tiles <= g_num_sms && !crowded ? TILE_SLIM : single_tiles <= g_num_sms ? TILE_SINGLE : pairs ? TILE_PAIR : TILE_WIDE;
    const bool pair = form == TILE_PAIR;
    const int tile_m = pair ? 2 * BM : BM, tile_n = form == TILE_SLIM ? TileShape<TILE_SLIM>::kN : form == TILE_SINGLE ? TileShape<TILE_SINGLE>::kN : TileShape<TILE_PAIR>::kN;

    static thread_local LargeParams gp;
    MapTable T(gp);
    int tiles = 0;
    for (int oi = 0; oi < n_ops; ++oi) {
        const GemmOp& op = ops[order[oi]];
        DevProblem& Q = gp.prob[oi];
        std::memset(&Q, 0, sizeof(Q));
        if (op.M < 1 || op.N < 1 || op.n_kseg < 1 || op.n_kseg > kMaxSeg || !op.C || op.ldc < 1) return ECOSPA_ERR_INVALID;
        if (op.M > INT32_MAX || op.N > INT32_MAX) return ECOSPA_ERR_INVALID;
        const bool swiglu = op.epi == EPI_SWIGLU;
        const int out_eb = op.out_f32 ? 4 : 2;
        if (!aligned16(op.C) || (op.ldc * out_eb) % 16) return ECOSPA_ERR_ALIGNMENT;
        if ((op.epi == EPI_GELU_ERF || op.epi == EPI_GELU_TANH || op.epi == EPI_DSWIGLU || swiglu) && (!op.C2 || !aligned16(op.C2)))
            return op.C2 ? ECOSPA_ERR_ALIGNMENT : ECOSPA_ERR_INVALID;
        if (swiglu && (!op.C3 || !aligned16(op.C3))) return op.C3 ? ECOSPA_ERR_ALIGNMENT : ECOSPA_ERR_INVALID;
        if (op.epi >= EPI_DGELU_ERF) {
            if (!op.H || (op.epi == EPI_DSWIGLU && !op.Hb)) return ECOSPA_ERR_INVALID;
            if (!aligned16(op.H) || (op.Hb && !aligned16(op.Hb)) || (op.ldh * 2) % 16) return ECOSPA_ERR_ALIGNMENT;
        }
        if (op.out_f32 && op.epi != EPI_STORE) return ECOSPA_ERR_UNSUPPORTED;
        if (op.bias && !aligned16(op.bias)) return ECOSPA_ERR_ALIGNMENT;
        Q.M = static_cast<int32_t>(op.M);
        Q.N = static_cast<int32_t>(op.N);
        Q.n_per_tile = swiglu ? tile_n / 2 : tile_n;
        Q.half1_n_off = swiglu ? 0 : tile_n / 2;
        Q.epi = op.epi;
        Q.out_f32 = op.out_f32;
        Q.accumulate = op.accumulate;
        Q.bias_f32 = op.bias_f32;
        Q.C = op.C; Q.C2 = op.C2; Q.C3 = op.C3;
        Q.bias = op.bias; Q.H = op.H; Q.Hb = op.Hb;
        Q.ldc = op.ldc; Q.ldh = op.ldh;
        for (int s = 0; s < op.n_kseg; ++s) {
            const KSegment& ks = op.seg[s];
            if (ks.K < 1 || ks.k_begin < 0 || ks.k_begin % BK) return ECOSPA_ERR_INVALID;
            // stored shapes must cover the logical (M, N, [k_begin, k_begin + K))
            const int64_t k_end = ks.k_begin + ks.K;
            const Stored& a = ks.a;
            // a range that stops before the end of the stored tensor must end on a k-block boundary
            if (k_end < (ks.a_mn ? a.rows : a.cols) && ks.K % BK) return ECOSPA_ERR_INVALID;
            if (ks.a_mn ? (a.rows < k_end || a.cols != op.M) : (a.rows != op.M || a.cols < k_end)) return ECOSPA_ERR_INVALID;
            int map = 0, how = 0;
            if ((st = operand_map(T, a, ks.a_mn, pair, 128, true, &map, &how)) != ECOSPA_OK) return st;
            Q.map_a[s] = static_cast<uint8_t>(map);
            Q.a_big[s] = how == FORM_BIG;
            Q.a_3d[s] = how == FORM_3D;
            for (int h = 0; h < 2; ++h) {
                const Stored& b = (swiglu && h == 1) ? ks.b[1] : ks.b[0];
                if (ks.b_mn ? (b.rows < k_end || b.cols != op.N) : (b.rows != op.N || b.cols < k_end)) return ECOSPA_ERR_INVALID;
                if ((st = operand_map(T, b, ks.b_mn, pair, std::max(64, tile_n / 2), tile_n == 256, &map, &how)) != ECOSPA_OK) return st;
                Q.map_b[s][h] = static_cast<uint8_t>(map);
                if (h == 0) {
                    Q.b_big[s] = how == FORM_BIG;
                    Q.b_3d[s] = how == FORM_3D;
                } else if ((how == FORM_BIG) != (Q.b_big[s] != 0) || (how == FORM_3D) != (Q.b_3d[s] != 0)) {
                    return ECOSPA_ERR_UNSUPPORTED;   // both halves take the same path
                }
            }
            Q.a_mn[s] = ks.a_mn;
            Q.b_mn[s] = ks.b_mn;
            Q.k_off[s] = static_cast<int32_t>(ks.k_begin);
            Q.kblocks += static_cast<int32_t>(ceil_div(ks.K, BK));
            Q.kb_end[s] = Q.kblocks;
        }
        // outputs leave through TMA tile stores (a reducing store when they are added to what C holds)
        {
            const bool wide = op.epi == EPI_STORE || op.epi == EPI_GELU_ERF || op.epi == EPI_GELU_TANH;
            void* outs[3] = {op.C, op.C2, op.C3};
            for (int o = 0; o < 3; ++o) {
                if (!outs[o]) continue;
                CUtensorMap* out = T.next();
                if (!out) return ECOSPA_ERR_UNSUPPORTED;
                if ((st = encode_out_map(out, outs[o], op.M, op.N, op.ldc, op.out_f32, wide)) != ECOSPA_OK) return st;
                Q.map_c[o] = static_cast<uint8_t>(T.add(Stored(), MapTable::kOutput));   // (never shared)
            }
        }
        for (int s2 = op.n_kseg; s2 < kMaxSeg; ++s2) Q.kb_end[s2] = Q.kblocks;
        Q.tiles_m = static_cast<int32_t>(ceil_div(op.M, tile_m));
        Q.tiles_n = static_cast<int32_t>(ceil_div(op.N, Q.n_per_tile));
        Q.tile_start = tiles;
        tiles += Q.tiles_m * Q.tiles_n;
    }
    gp.head.n_problems = n_ops;
    gp.head.total_tiles = tiles;
    gp.head.status = dev->status_ptr;
    gp.head.side.n_jobs = gp.head.side.whole = 0;
    if (side && side->n_jobs > 0) gp.head.side = *side;
    gp.head.wait_limit_ns = g_wait_limit_ns.load(std::memory_order_relaxed);
    const int workers = pair ? std::min(tiles, g_max_pairs) : std::min(tiles, g_num_sms);
    build_schedule(gp, workers);
    const cudaError_t e = pair ? launch_smallest_form<TILE_PAIR>(gp, T.n, workers, stream)
                          : form == TILE_SLIM ? launch_smallest_form<TILE_SLIM>(gp, T.n, workers, stream)
                          : form == TILE_SINGLE ? launch_smallest_form<TILE_SINGLE>(gp, T.n, workers, stream)
                                                : launch_smallest_form<TILE_WIDE>(gp, T.n, workers, stream);
    if (e != cudaSuccess) {
        set_cuda_error(e, "gemm_kernel launch");
        cudaGetLastError();
        return ECOSPA_ERR_CUDA;
    }
    return check_launch("gemm_kernel");
}

int* engine_status_ptr(ecospa_status_t* st) {
    DeviceState* dev = gemm_setup(st);
    return dev ? dev->status_ptr : nullptr;
}
int engine_num_sms() {
    ecospa_status_t st;
    DeviceState* dev = gemm_setup(&st);
    return dev ? dev->num_sms : 0;
}
unsigned long long engine_wait_limit_ns() { return g_wait_limit_ns.load(std::memory_order_relaxed); }

int gemm_resident_pairs() {
    ecospa_status_t st;
    DeviceState* dev = gemm_setup(&st);
    if (!dev) return -1;
    return g_pair_mode ? dev->max_pairs : 0;
}

}  // namespace ecospa

extern "C" ecospa_status_t ecospa_device_status(void* stream, int32_t* code) {
    if (!code) return ECOSPA_ERR_INVALID;
    ecospa_status_t st;
    ecospa::DeviceState* dev = ecospa::gemm_setup(&st);
    if (!dev) return st;
    cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    int v = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&v, dev->status_ptr, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) {
        ecospa::set_cuda_error(e, "ecospa_device_status");
        return ECOSPA_ERR_CUDA;
    }
    *code = v;
    if (v != 0) {
        cudaMemset(dev->status_ptr, 0, sizeof(int));
        return ECOSPA_ERR_TIMEOUT;
    }
    return ECOSPA_OK;
}

// Number of CTA pairs the GEMM engine runs at once on the current device (0 = pair mode off).
extern "C" int32_t ecospa_gemm_resident_pairs(void) { return ecospa::gemm_resident_pairs(); }

extern "C" ecospa_status_t ecospa_set_device_wait_limit_ns(uint64_t ns) {
    if (ns == 0) return ECOSPA_ERR_INVALID;
    ecospa::g_wait_limit_ns.store(ns, std::memory_order_relaxed);
    return ECOSPA_OK;
}

// Linear layers with few token rows: Y[rows][out] = act(X[rows][in] * Wm[out][in]^T + bias) (+ residual), straight
// from the packed weight (Sec. 2, Fig. 2 bottom of the ELSA paper), one launch for one layer or for many.
//
// A layer of one or a few images has too few 256-row tiles to occupy the SM pairs of the persistent kernels, and what
// it pays for is latency: the launch of the kernel that rebuilds the weight image, a persistent kernel's set-up, one
// long reduction per tile.  Here
//   * a call of one layer at 1:4 or 2:4 has the weight tile expanded on the way to shared memory by eight warps that read
//     the packed values and index words, so that there is no image and no second launch (the code takes every level, and
//     the dense shared weight for the masked form, where the variant is forced; by itself the library brings an image, see
//     the rule in elsa_api.cu); the dense level's tile comes by TMA, and so do the images that the layers of a table and
//     of a chained block bring along (one launch builds those of a whole call);
//   * a CTA computes one tile of 128 rows x 64 features and leaves; two CTAs fit an SM, so that one's set-up and
//     epilogue run under the other's tile, or the next kernel's set-up under this one's;
//   * where the tiles alone leave SMs idle, the reduction is cut into 2, 4 or 8 ranges, one CTA of a cluster each:
//     every CTA sends the rows of its fp32 sums to the CTA that owns them, and each owner adds its rows in rank order
//     (deterministic), applies bias, activation and residual, which it has asked for by then, and rounds once;
//   * the sums go as bulk copies between the CTAs' shared memories, whose bytes the owner's barrier counts, in a chain and in a call
//     of its own on a dense weight (1024 -> 1024 at 4:4, 49 rows, 6.9 -> 6.1 us; one-image encoder 500 -> 492), elsewhere as stores into
//     the other CTA's memory and a cluster barrier: that is less code, and where an image kernel runs between any two of
//     these no cache holds it (1536 -> 384 at 1:8, 197 rows, image included, bulk copies 7.5, stores 7.0 us);
//   * a call that knows the weights to be older than its own first kernel (the chained block) has their first tiles
//     fetched before the predecessor kernel has ended (`early`): only X and the outputs wait for it;
//   * in a chain each launch has the next linear's weight brought into L2 (`ahead`): a model's weights do not stay there
//     from one call to the next (one-image encoder 486 -> 476 us).
// Measured back to back on 197 rows (us, weight image + one-CTA-per-tile GEMM before, this kernel after): 768 -> 768 at
// 2:4 6.9 -> 6.4, 768 -> 2304 at 2:4 8.2 -> 7.7, 3072 -> 768 at 2:4 15.4 -> 10.6, at 4:4 11.6 -> 6.9.  The expansion
// is repeated for every 128 rows and bound by its loads' latency and its instructions: at 788 rows and 2:4 the image
// kernel and a GEMM that reads it take 10.9 us where this one takes 20.
//
// Warps: 0 TMA producer, 1 MMA issuer (tcgen05, M = 128), 2-9 expansion, then epilogue, 10-11 only barriers.

#include <atomic>
#include <type_traits>

#include "elsa_tc_common.cuh"
#include "elsa_pack_device.cuh"

namespace elsa {
namespace {

constexpr int kTileM = 128;
constexpr int kTileN = 64;
constexpr int kTileK = 64;                 // one 128-byte swizzle row
constexpr int kWorkers = 8;                // expansion / epilogue warps
// Registers are allocated for four warps at a time: ten warps cost what twelve do, and two CTAs per SM leave 80
// registers to each thread of twelve.
constexpr int kSmallThreads = 12 * 32;
constexpr int kXBytes = kTileM * kTileK * 2;
constexpr int kWBytes = kTileN * kTileK * 2;
constexpr int kStageBytes = kXBytes + kWBytes;
constexpr int kStagesMax = 4;
constexpr int kStagesSplit = 3;
constexpr int kHalfN = kTileN / 2;         // columns of an epilogue warp
constexpr int kPitch = kHalfN + 4;         // floats of a row of a warp's sums: 16-byte accesses of 8 rows fall on 32 banks
constexpr int kSumBytes = 2 * kTileM * kPitch * 4;
constexpr int kSplitsMax = 8;
constexpr int kAheadUnits = 512;           // of 16 bytes in one request for the next linear's weight
constexpr int kSmallGroupMax = 72;         // layers per launch (kernel parameters are limited to 32 KB)

// Two CTAs per SM need at most 113 KB each.  With one range the sums take the place of the stages; with several those
// that arrive have their own, since another CTA of the cluster may send its sums while this one's MMAs still read.
constexpr int small_smem(bool split)
{
    return (split ? kStagesSplit * kStageBytes + kSumBytes : kStagesMax * kStageBytes) + 256 /* barriers */ + 1024 /* alignment */;
}

enum WeightSource { SRC_DENSE = 0, SRC_PACKED = 1, SRC_MASK = 2 };

struct alignas(64) SmallLayer {
    CUtensorMap map_x;
    CUtensorMap map_w;            // SRC_DENSE
    const uint16_t* w;            // packed values, or the dense shared weight (SRC_MASK)
    const uint32_t* idx;
    const uint16_t* bias;
    const uint16_t* residual;
    uint16_t* Y;
    int rows, in, out, N, M, source;
    int tiles_n, tile_begin, k_blocks, words_per_row, act;
};

template <int kMax>
struct SmallGroup {
    SmallLayer layer[kMax];
    int n_layers;
    int splits;                   // CTAs of a cluster = ranges of the reduction
    int stages;
    int early;
    int first_pass;               // of the epilogue: 0 the rehearsal, 1 the real one
    uint32_t idesc;
    uint32_t* dev_status;
    const void* ahead;            // what the call's next linear reads as its weight: brought into L2 meanwhile
    uint32_t ahead_units;         // of 16 bytes
};

__device__ __forceinline__ void bulk_prefetch_l2(const void* src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void named_barrier_workers() { asm volatile("bar.sync 1, %0;" ::"n"(kWorkers * 32) : "memory"); }

// Copies shared memory of this CTA into another one of the cluster, the bytes counted on an mbarrier there.
__device__ __forceinline__ void bulk_send(uint32_t dst_cluster, uint32_t src, uint32_t bytes, uint32_t bar_cluster)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst_cluster), "r"(src),
                 "r"(bytes), "r"(bar_cluster)
                 : "memory");
}

// The expansion of the K blocks kb0..kb1 by two groups of four warps that take turns, kAhead K blocks at a time: one
// group's loads are in flight while the other expands.  (One group alone pays an L2 round trip per turn, however early
// it asks: the proxy fence that publishes a tile to the MMA also waits for the loads in flight.)  A thread has the rows
// row0 + 16 i of the weight tile and one 16-byte unit of the 64 k; load(row, unit) returns what it read, finish(raw,
// unit) the expanded unit.
template <int kAhead, typename Raw, typename Load, typename Finish>
__device__ __forceinline__ bool expand_range(int kb0, int kb1, int stages, uint32_t smem_base, uint32_t full_bar, uint32_t empty_bar,
                                             int n0, int out, int in, volatile uint32_t* abort_flag, uint32_t* dev_status, Load load,
                                             Finish finish)
{
    constexpr int kRows = kTileN / 16;
    const int tid = (int)threadIdx.x - 64;
    const int row0 = (tid & 127) >> 3, unit = tid & 7;
    Raw raw[kAhead][kRows];
    for (int kbase = kb0 + kAhead * (tid >> 7); kbase < kb1; kbase += 2 * kAhead) {
        const int count = min(kAhead, kb1 - kbase);
#pragma unroll
        for (int d = 0; d < kAhead; ++d) {
            const int u = (kbase + d) * (kTileK / 8) + unit;
#pragma unroll
            for (int i = 0; i < kRows; ++i)
                if (d < count && n0 + row0 + 16 * i < out && 8 * u < in) raw[d][i] = load(n0 + row0 + 16 * i, u);
        }
#pragma unroll
        for (int d = 0; d < kAhead; ++d) {
            if (d >= count) break;
            const int turn = (kbase + d - kb0) / stages, stage = (kbase + d - kb0) - turn * stages;
            bool ok = mbar_wait(empty_bar + 8 * stage, (turn & 1) ^ 1, abort_flag, dev_status, 41);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) return false;
            const uint32_t tile = smem_base + (uint32_t)(stage * kStageBytes) + kXBytes;
            const int u = (kbase + d) * (kTileK / 8) + unit;
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                const int r = row0 + 16 * i;
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (n0 + r < out && 8 * u < in) v = finish(raw[d][i], u);
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(tile + (uint32_t)(r * 128) + (uint32_t)((unit ^ (r & 7)) << 4)),
                             "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                             : "memory");
            }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if ((threadIdx.x & 31) == 0)
            for (int d = 0; d < count; ++d) mbar_arrive(full_bar + 8 * ((kbase + d - kb0) % stages));
    }
    return true;
}

struct DenseRaw { uint4 a, b; };
struct NoRaw { int row; };

// kBulk: how the sums of a cut reduction go to their owners, see above.
template <bool kBf16, int kMax, bool kBulk>
__global__ void __launch_bounds__(kSmallThreads, 2) linear_small_kernel(const __grid_constant__ SmallGroup<kMax> p)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int splits = p.splits;
    const bool split = splits > 1;
    const int rank = split ? (int)cluster_ctarank() : 0;
    const int tile_all = (int)blockIdx.x / splits;

    int cur = 0;
    if constexpr (kMax > 1) {
        int hi = p.n_layers - 1;
        while (cur < hi) {
            const int mid = (cur + hi + 1) >> 1;
            if (p.layer[mid].tile_begin <= tile_all) cur = mid; else hi = mid - 1;
        }
    }
    const SmallLayer& L = p.layer[cur];
    const int tile = tile_all - L.tile_begin;
    const int m0 = (tile / L.tiles_n) * kTileM, n0 = (tile % L.tiles_n) * kTileN;
    const int kb0 = L.k_blocks * rank / splits, kb1 = L.k_blocks * (rank + 1) / splits;
    const bool expand = kMax == 1 && L.source != SRC_DENSE;      // a group's weights are all dense or images

    const int sums_off = split ? p.stages * kStageBytes : 0;
    const int bar_off = split ? sums_off + kSumBytes : p.stages * kStageBytes;
    const uint32_t full_bar = smem_base + (uint32_t)bar_off;
    const uint32_t empty_bar = full_bar + 8 * kStagesMax;
    const uint32_t done_bar = empty_bar + 8 * kStagesMax;
    const uint32_t sums_bar = done_bar + 8;       // kBulk: the sums of this CTA's rows: its own warps' arrivals, the others' bytes
    volatile uint32_t* tmem_holder = reinterpret_cast<volatile uint32_t*>(smem_gen + bar_off + 16 * kStagesMax + 16);
    const int slice = kTileM / splits;            // rows each CTA of the cluster finishes
    volatile uint32_t* abort_flag = tmem_holder + 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(full_bar + 8 * s, expand ? 1 + kWorkers / 2 : 1);
            mbar_init(empty_bar + 8 * s, 1);
        }
        mbar_init(done_bar, 1);
        if constexpr (kBulk) {
            mbar_init(sums_bar, 1 + kWorkers);
            mbar_arrive_expect_tx(sums_bar, (uint32_t)((splits - 1) * slice * 2 * kPitch * 4));
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
    }
    if (warp == 1) tmem_alloc(smem_base + (uint32_t)(bar_off + 16 * kStagesMax + 16), kTileN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    // A CTA of the cluster writes into another's shared memory only once that one runs (first phase of the cluster's
    // barrier), and leaves only when what it sent has arrived (second phase).
    if (split) cluster_arrive();

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        const bool elected = elect_one();
        const uint32_t tx = (uint32_t)(kXBytes + (expand ? 0 : kWBytes));
        const int first = kb1 - kb0 < p.stages ? kb1 - kb0 : p.stages;      // stages filled without a wait
        if (!p.early) {
            pdl_wait_for_predecessors();
            pdl_release_successors();
        }
        if (elected)
            for (int s = 0; s < first; ++s) {
                mbar_arrive_expect_tx(full_bar + 8 * s, tx);
                if (!expand) tma_load_2d(smem_base + (uint32_t)(s * kStageBytes) + kXBytes, &L.map_w, full_bar + 8 * s, (kb0 + s) * kTileK, n0);
            }
        __syncwarp();
        if (p.early) {
            pdl_wait_for_predecessors();
            pdl_release_successors();
        }
        if (elected)
            for (int s = 0; s < first; ++s)
                tma_load_2d(smem_base + (uint32_t)(s * kStageBytes), &L.map_x, full_bar + 8 * s, (kb0 + s) * kTileK, m0);
        __syncwarp();
        int stage = 0;
        uint32_t phase = 0;
        for (int kb = kb0 + first; kb < kb1; ++kb) {
            bool ok = mbar_wait(empty_bar + 8 * stage, phase, abort_flag, p.dev_status, 42);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            if (elected) {
                const uint32_t dst = smem_base + (uint32_t)(stage * kStageBytes);
                mbar_arrive_expect_tx(full_bar + 8 * stage, tx);
                tma_load_2d(dst, &L.map_x, full_bar + 8 * stage, kb * kTileK, m0);
                if (!expand) tma_load_2d(dst + kXBytes, &L.map_w, full_bar + 8 * stage, kb * kTileK, n0);
            }
            __syncwarp();
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
        if (split) { cluster_wait(); cluster_arrive(); cluster_wait(); }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer (whole warp, one elected lane issues)
        const uint32_t elected = elect_one() ? 1u : 0u;
        const uint32_t d_tmem = __reduce_or_sync(0xFFFFFFFFu, tmem_base);
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int kb = kb0; kb < kb1; ++kb) {
            ok = mbar_wait(full_bar + 8 * stage, phase, abort_flag, p.dev_status, 43);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint32_t x_addr = smem_base + (uint32_t)(stage * kStageBytes);
            const uint64_t a_desc = smem_desc_k_major_sw128(x_addr);
            const uint64_t b_desc = smem_desc_k_major_sw128(x_addr + kXBytes);
#pragma unroll
            for (int k = 0; k < kTileK / 16; ++k)
                umma_f16_if(d_tmem, a_desc + (uint64_t)(2 * k), b_desc + (uint64_t)(2 * k), p.idesc, (uint32_t)(kb != kb0 || k != 0), elected);
            umma_commit_if(empty_bar + 8 * stage, elected);
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit_if(done_bar, elected);
        __syncwarp();
        if (split) { cluster_wait(); cluster_arrive(); cluster_wait(); }
    } else if (warp >= 2 + kWorkers) {
        if (warp == 2 + kWorkers && p.ahead != nullptr && elect_one()) {
            // a chained block's weights do not stay in L2 from one call to the next: each CTA asks for its share of the next ones
            pdl_wait_for_predecessors();
            const uint32_t share = (p.ahead_units + gridDim.x - 1) / gridDim.x, end = min(p.ahead_units, share * (blockIdx.x + 1));
            for (uint32_t at = share * blockIdx.x; at < end; at += kAheadUnits)
                bulk_prefetch_l2(static_cast<const uint4*>(p.ahead) + at, 16u * min((uint32_t)kAheadUnits, end - at));
        }
        __syncwarp();
        if (split) { cluster_wait(); cluster_arrive(); cluster_wait(); }
    } else {
        // ------------------------------------------------ expansion, then epilogue
        if (!p.early) pdl_wait_for_predecessors();
        bool ok = true;
        if constexpr (kMax == 1) if (expand) {
            const uint16_t* w = L.w;
            const uint32_t* idx = L.idx;
            const int N = L.N, in = L.in, wpr = L.words_per_row;
            auto run = [&](auto ahead, auto raw_type, auto load, auto finish) {
                return expand_range<decltype(ahead)::value, decltype(raw_type)>(kb0, kb1, p.stages, smem_base, full_bar, empty_bar, n0, L.out,
                                                                               in, abort_flag, p.dev_status, load, finish);
            };
            if (L.source == SRC_PACKED) {
                const int vpr = in / L.M * N;
#define ELSA_EXPAND_PACKED(M, NC)                                                                                              \
    ok = run(std::integral_constant<int, NC ? 2 : 1>{}, PackedUnit{},                                                          \
             [&](int row, int u) { return load_packed_unit<M, NC>(w + (size_t)row * vpr, idx + (size_t)row * wpr, N, u); },    \
             [&](const PackedUnit& raw, int) { return expand_packed_unit<M, NC>(raw, N); })
                if (L.M == 8) {
                    if (N == 1) ELSA_EXPAND_PACKED(8, 1);
                    else if (N == 2) ELSA_EXPAND_PACKED(8, 2);
                    else if (N == 4) ELSA_EXPAND_PACKED(8, 4);
                    else ELSA_EXPAND_PACKED(8, 0);
                } else if (L.M == 4) {
                    if (N == 1) ELSA_EXPAND_PACKED(4, 1);
                    else if (N == 2) ELSA_EXPAND_PACKED(4, 2);
                    else ELSA_EXPAND_PACKED(4, 0);
                } else {
                    ok = run(std::integral_constant<int, 1>{}, NoRaw{}, [&](int row, int) { return NoRaw{row}; },
                             [&](const NoRaw& raw, int u) { return expand_unit16(w + (size_t)raw.row * vpr, idx + (size_t)raw.row * wpr, N, u); });
                }
#undef ELSA_EXPAND_PACKED
            } else if (L.M == 16) {
                ok = run(std::integral_constant<int, 1>{}, DenseRaw{},
                         [&](int row, int u) {
                             const uint4* g = reinterpret_cast<const uint4*>(w + (size_t)row * in + (size_t)(u >> 1) * 16);
                             return DenseRaw{__ldcg(g), __ldcg(g + 1)};
                         },
                         [&](const DenseRaw& raw, int u) { return mask_unit<16>(raw.a, raw.b, u & 1, N); });
            } else {
                const bool eight = L.M == 8;
                ok = run(std::integral_constant<int, 2>{}, uint4{},
                         [&](int row, int u) { return __ldcg(reinterpret_cast<const uint4*>(w + (size_t)row * in + (size_t)u * 8)); },
                         [&](const uint4& raw, int) { return eight ? mask_unit<8>(raw, raw, 0, N) : mask_unit<4>(raw, raw, 0, N); });
            }
        }
        if (p.early) pdl_wait_for_predecessors();     // before the residual is read or Y written
        const int q = warp & 3, half = (warp - 2) >> 2;
        // What the finished rows need besides the sums is asked for ahead of them.
        constexpr int kUnits = kTileN / 8, kRowsAStep = kWorkers * 32 / kUnits;
        const int tid = (int)threadIdx.x - 64;
        const int col_l = (tid % kUnits) * 8, col = n0 + col_l;      // the same for all of a thread's units
        uint4 bw = make_uint4(0u, 0u, 0u, 0u), rw = bw;
        if (L.bias != nullptr && col < L.out) bw = __ldg(reinterpret_cast<const uint4*>(L.bias + col));
        const uint16_t* residual = L.residual;
        const int rows_here = col < L.out ? min(slice, L.rows - m0 - rank * slice) : 0;      // to finish; none if it is not positive
        {
            const int row = m0 + rank * slice + tid / kUnits;
            if (residual != nullptr && tid / kUnits < rows_here) rw = *reinterpret_cast<const uint4*>(residual + (size_t)row * L.out + col);
        }
        // The sums of 32 rows x 32 columns a warp lie [half][row][pitch]; those that come from CTA s of the cluster at
        // s * slice rows of either half.
        const uint32_t inbox = smem_base + (uint32_t)sums_off;
        const float* sums = reinterpret_cast<const float*>(smem_gen + sums_off) + (size_t)(col_l / kHalfN * kTileM) * kPitch + col_l % kHalfN;
        // In a chain the first pass is a rehearsal: while the loads and MMAs are under way it runs the last part's instructions and
        // stores nothing (what it reads of the sums is whatever lies there, stages that TMA is filling included, and goes nowhere).
        // In a chain of kernels their code is in none of the SM's caches, and fetched when it is needed it took longer than it ran:
        // one-image encoder of DeiT-B 492 -> 486 us; for the same reason the loops here are not unrolled.  Calls of one's own keep
        // the code and only pay for the pass: 1536 -> 384 at 4:4, 49 rows, 5.6 us with it, 4.9 without.
#pragma unroll 1
        for (int real = p.first_pass; real < 2; ++real) {
            if (real) {
                ok = ok && mbar_wait(done_bar, 0, abort_flag, p.dev_status, 44);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (split) cluster_wait();
                if (ok) {
                    tc_fence_after();
                    const int row = q * 32 + lane, to = row / slice;
                    uint32_t r[32];
                    tmem_ld_32x32b_x32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * kHalfN), r);
                    tmem_wait_ld();
                    tc_fence_before();
                    const uint32_t in_owner = inbox + (uint32_t)((half * kTileM + rank * slice + row % slice) * kPitch * 4);
                    if constexpr (kBulk) {
                        // rows of this CTA go where they are added, the others' to the stages (no MMA reads them any more) and from
                        // there to their CTA as one copy for each
                        const uint32_t outbox = smem_base + (uint32_t)(half * kTileM * kPitch * 4);
                        const uint32_t dst = to == rank ? in_owner : outbox + (uint32_t)(row * kPitch * 4);
#pragma unroll
                        for (int v = 0; v < 8; ++v)
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (uint32_t)(16 * v)), "r"(r[4 * v]),
                                         "r"(r[4 * v + 1]), "r"(r[4 * v + 2]), "r"(r[4 * v + 3])
                                         : "memory");
                        if (split) fence_proxy_async_smem();
                        __syncwarp();
                        if (split) {
                            const int run = min(slice, 32);      // a warp's rows for one CTA
                            if (to != rank && lane % run == 0)
                                bulk_send(mapa_shared(in_owner, (uint32_t)to), outbox + (uint32_t)(row * kPitch * 4),
                                          (uint32_t)(run * kPitch * 4), mapa_shared(sums_bar, (uint32_t)to));
                        }
                        if (lane == 0) mbar_arrive(sums_bar);
                        ok = mbar_wait(sums_bar, 0, abort_flag, p.dev_status, 45);
                        ok = __all_sync(0xFFFFFFFFu, ok);
                    } else {
                        const uint32_t dst = split ? mapa_shared(in_owner, (uint32_t)to) : in_owner;
#pragma unroll
                        for (int v = 0; v < 8; ++v)
                            asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (uint32_t)(16 * v)), "r"(r[4 * v]),
                                         "r"(r[4 * v + 1]), "r"(r[4 * v + 2]), "r"(r[4 * v + 3])
                                         : "memory");
                    }
                }
                if (split) cluster_arrive();
                if constexpr (!kBulk) {
                    __syncwarp();
                    if (split) cluster_wait();
                    else named_barrier_workers();
                }
            }
            if (ok) {
#pragma unroll 1
                for (int row_l = real ? tid / kUnits : slice - 1; row_l < (real ? rows_here : slice); row_l += kRowsAStep) {
                    const int row = m0 + rank * slice + row_l;
                    if (real && row_l >= kRowsAStep && residual != nullptr)
                        rw = *reinterpret_cast<const uint4*>(residual + (size_t)row * L.out + col);
                    float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
                    for (int s = 0; s < splits; ++s) {
                        const float4* src = reinterpret_cast<const float4*>(sums + (size_t)(s * slice + row_l) * kPitch);
                        const float4 x = src[0], y = src[1];
                        a[0] += x.x; a[1] += x.y; a[2] += x.z; a[3] += x.w;
                        a[4] += y.x; a[5] += y.y; a[6] += y.z; a[7] += y.w;
                    }
                    const uint32_t b[4] = {bw.x, bw.y, bw.z, bw.w}, r[4] = {rw.x, rw.y, rw.z, rw.w};
                    uint32_t o[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float2 bv = raw2_to_float2<kBf16>(b[j]);
                        a[2 * j] += bv.x;
                        a[2 * j + 1] += bv.y;
                    }
                    if (L.act == 1) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float2 g = gelu_pair(a[2 * j], a[2 * j + 1]);
                            a[2 * j] = g.x;
                            a[2 * j + 1] = g.y;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float2 rv = raw2_to_float2<kBf16>(r[j]);
                        o[j] = pack2<kBf16>(a[2 * j] + rv.x, a[2 * j + 1] + rv.y);
                    }
                    if (real) *reinterpret_cast<uint4*>(L.Y + (size_t)row * L.out + col) = make_uint4(o[0], o[1], o[2], o[3]);
                }
            }
        }
        if (kBulk && split) cluster_wait();
    }

    // ------------------------------------------------ teardown
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (*abort_flag)
            for (int i = 0; i < 200; ++i) __nanosleep(10000);     // copies and MMAs in flight land first
        tc_fence_after();
        tmem_dealloc(tmem_base, kTileN);
    }
}

template <bool kBf16, int kMax, bool kBulk>
elsa_status launch_small(const SmallJob* jobs, int n, int splits, bool early, uint32_t* dev_status, cudaStream_t stream, const DeviceInfo& dev)
{
    SmallGroup<kMax> g;      // on the stack: several threads may launch at once
    int tile_begin = 0;
    for (int i = 0; i < n; ++i) {
        const SmallJob& j = jobs[i];
        SmallLayer& L = g.layer[i];
        L.w = j.w; L.idx = j.idx; L.bias = j.bias; L.residual = j.residual; L.Y = j.Y;
        L.rows = j.rows; L.in = j.in; L.out = j.out; L.N = j.N; L.M = j.M; L.act = j.act;
        L.source = j.N == j.M ? SRC_DENSE : j.masked ? SRC_MASK : SRC_PACKED;
        L.tiles_n = (j.out + kTileN - 1) / kTileN;
        L.tile_begin = tile_begin;
        tile_begin += ((j.rows + kTileM - 1) / kTileM) * L.tiles_n;
        L.k_blocks = (j.in + kTileK - 1) / kTileK;
        L.words_per_row = (int)index_words_per_row(j.in, j.N, j.M);
        elsa_status st;
        if ((st = make_map_2d(&L.map_x, j.X, (uint64_t)j.in, (uint64_t)j.rows, kTileK, kTileM, CU_TENSOR_MAP_SWIZZLE_128B, "X")) != ELSA_OK)
            return st;
        if (L.source == SRC_DENSE &&
            (st = make_map_2d(&L.map_w, j.w, (uint64_t)j.in, (uint64_t)j.out, kTileK, kTileN, CU_TENSOR_MAP_SWIZZLE_128B, "W")) != ELSA_OK)
            return st;
    }
    constexpr uint32_t fmt = kBf16 ? 1u : 0u;
    g.n_layers = n;
    g.splits = splits;
    g.stages = splits > 1 ? kStagesSplit : kStagesMax;
    g.early = early ? 1 : 0;
    g.first_pass = n == 1 && jobs[0].chained ? 0 : 1;
    g.idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(kTileN >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
    g.dev_status = dev_status;
    g.ahead = n == 1 ? jobs[0].ahead : nullptr;
    g.ahead_units = n == 1 ? (uint32_t)(jobs[0].ahead_bytes / 16) : 0;

    auto kernel = linear_small_kernel<kBf16, kMax, kBulk>;
    constexpr int kSmemMost = small_smem(true) > small_smem(false) ? small_smem(true) : small_smem(false);
    static std::atomic<bool> attr_set[64];
    const int slot = dev.device & 63;
    if (!attr_set[slot].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMost) != cudaSuccess) {
            cudaError_t e = cudaGetLastError();
            return fail(ELSA_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
        }
        attr_set[slot].store(true, std::memory_order_release);
    }
    ProfileScope scope(ELSA_KERNEL_LINEAR_SMALL, stream);
    cudaError_t e = launch_pdl(kernel, dim3((unsigned)(tile_begin * splits)), dim3(kSmallThreads), (size_t)small_smem(splits > 1), stream,
                               (unsigned)splits, g);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(ELSA_ERR_CUDA, "launch of linear_small failed: %s", cudaGetErrorString(e));
    }
    return launched("linear_small");
}

}  // namespace

int linear_small_group_max() { return kSmallGroupMax; }

// One CTA per SM: a second wave, or two CTAs sharing an SM, costs more than the shorter ranges give (768 -> 2304 on 197
// rows at 4:4: 5.3 us with 144 CTAs, 11.9 with 288).  A range keeps at least two K blocks.
int linear_small_splits(const SmallJob* jobs, int n, int sm_count)
{
    long long tiles = 0;
    int k_least = 1 << 30;
    for (int i = 0; i < n; ++i) {
        tiles += (long long)((jobs[i].rows + kTileM - 1) / kTileM) * ((jobs[i].out + kTileN - 1) / kTileN);
        const int kb = (jobs[i].in + kTileK - 1) / kTileK;
        if (kb < k_least) k_least = kb;
    }
    int splits = 1;
    while (splits < kSplitsMax && tiles * splits * 2 <= sm_count && k_least >= 4 * splits) splits *= 2;
    return splits;
}

elsa_status launch_linear_small_group(const SmallJob* jobs, int n, int splits, bool early, elsa_dtype dtype, uint32_t* dev_status,
                                      cudaStream_t stream)
{
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    if (n < 1 || n > kSmallGroupMax) return fail(ELSA_ERR_SHAPE, "a grouped launch carries 1 to %d layers, got %d", kSmallGroupMax, n);
    for (int i = 0; n > 1 && i < n; ++i)
        if (jobs[i].N != jobs[i].M) return fail(ELSA_ERR_NM, "layer %d of a grouped launch is packed (%d:%d)", i, jobs[i].N, jobs[i].M);
    const bool bulk = n == 1 && (jobs[0].chained || (jobs[0].N == jobs[0].M && !jobs[0].after_image));
#define ELSA_SMALL(MAX, BULK)                                                                                   \
    (dtype == ELSA_BF16 ? launch_small<true, MAX, BULK>(jobs, n, splits, early, dev_status, stream, dev)        \
                        : launch_small<false, MAX, BULK>(jobs, n, splits, early, dev_status, stream, dev))
    if (n > 1) return ELSA_SMALL(kSmallGroupMax, false);
    return bulk ? ELSA_SMALL(1, true) : ELSA_SMALL(1, false);
#undef ELSA_SMALL
}

}  // namespace elsa

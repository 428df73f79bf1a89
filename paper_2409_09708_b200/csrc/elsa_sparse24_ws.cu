// N:M sparse linear (N <= 2) on the 2:4 sparse MMA with the weight held in tensor memory.
//
// Same product as elsa_sparse24_pair.cu (Sec. 2, Fig. 2 bottom of the ELSA paper, on the 2-of-4
// re-encoding of the packed weight).  That kernel streams the compressed weight tile and its metadata
// through shared memory again for every tile of token rows, and at the sparse MMA rate the weight and
// activation bytes together exceed what shared memory can deliver per cycle.  Here the weight does
// not move: a CTA pair owns one block of 256 output features of a layer for the whole layer.  Its
// 2-of-4 values (in/4 columns) and metadata (in/32 columns) are written once into the tensor memory
// of the two CTAs and every tcgen05.mma.sp reads its A operand from there; shared memory carries
// activations only.  What is left of tensor memory holds TWO accumulators of `nt` token rows each
// (144 for in = 768), so the epilogue of one tile runs under the MMAs of the next.  Narrow MMAs only
// pay because the issuing lane is predicated inside the instruction's own asm block: a branch around
// each tcgen05.mma costs the issuing warp about 80 cycles per instruction, the predicated form under
// 40, and a sparse MMA over 144 token rows lasts 72.
//
// Schedule of a layer over P pairs: F = ceil(out / 256) feature blocks, G = P / F row groups.  Pair p
// takes feature block p % F and the row tiles g, g + G, g + 2G, ... with g = p / F, so the F pairs
// of a group read the same activation rows at about the same time (one fetch from HBM, the rest from
// L2).  Pairs beyond G * F sit the layer out.  A launch may carry several layers; each pair walks
// them in order, reloading its weight block at every layer.
//
// Per CTA: warp 0 TMA producer for this CTA's half of the activation rows; warp 1 tensor-memory
// allocation and, in the leader, MMA issue; twelve epilogue warps (three per tensor-memory lane
// quarter, each with its own run of token columns) write the weight block into tensor memory at the
// start of a layer and run the epilogue.  The accumulator is transposed (lanes are features, columns
// are token rows) and Y is row-major, so the epilogue has to turn a lane's column pair into a row's
// feature run.  stmatrix with .trans does that in one instruction per 8 x 32 outputs if lane t of a
// quarter holds feature 8 * (t % 4) + t / 4 of its 32, so lane t writes that feature's row into tensor memory.
//
// The weight block is made from the packed weight itself: a lane expands its feature's row to two values per chunk of 4 and
// metadata on the way to tensor memory, 128 k at a time.  As an image the weight cost a launch of 2 to 3 us ahead of the layer
// and a trip through L2 for work that is a few hundred instructions a lane here, once a layer: 4925 x 768 -> 3072 at 2:4 20.4
// (on the streaming kernel, image included) -> 17.1 us, 3152 rows 16.0 -> 14.1; the linears of a DeiT-B block at 12608
// rows in a table 145 -> 143.  Only the masked form, whose dense shared weight would be ranked again by every row group, brings an image
// (SP24_PERMUTED form of launch_images: rows in the lanes' order).  Waits are bounded as in the other kernels.

#include <atomic>
#include <mutex>
#include <type_traits>

#include "elsa_sp24_device.cuh"
#include "elsa_tc_common.cuh"

namespace elsa {
namespace {

constexpr int kFeatPerCta = 128;   // weight rows per CTA = TMEM lanes
constexpr int kPairFeat = 256;     // MMA M over the pair
constexpr int kBlockK = 128;       // granularity of `in` (one metadata block)
constexpr int kStageK = 256;       // logical K per pipeline stage: eight MMAs per barrier round trip
constexpr int kSpUmmaK = 32;
constexpr int kNumAccum = 2;
constexpr int kTmemCols = 512;
constexpr int kMaxIn = 1024;       // in / 4 + in / 32 + 2 * nt columns must fit 512
constexpr int kMaxStages = 8;
constexpr int kEpiParts = 3;       // epilogue warps per TMEM lane quarter
constexpr int kEpiWarps = 4 * kEpiParts;
constexpr int kThreads = 64 + kEpiWarps * 32;
constexpr int kStepCols = 16;      // token rows per tcgen05.ld / pair of stmatrix
constexpr int kMaxSteps = 4;       // steps per epilogue warp and tile
constexpr int kMaxRowTile = kStepCols * kMaxSteps * kEpiParts;   // 192 token rows per pair tile (MMA N)
constexpr int kStagingBytes = kMaxSteps * kStepCols * 64;        // per epilogue warp: rows of 32 features
constexpr int kStagingTotal = kEpiWarps * kStagingBytes;
constexpr int kBarrierBytes = 512;

// The level of a packed weight.
enum WsLevel : uint8_t { LEVEL_1_4, LEVEL_2_4, LEVEL_1_8, LEVEL_2_8, LEVEL_1_16, LEVEL_2_16 };

struct alignas(64) WsLayer {
    CUtensorMap map_x, map_y, map_run;   // map_y: one step of 16 token rows, map_run: a warp's whole run of them
    // kImage: 2-of-4 values [out rounded up to 32][in / 2], rows in the permuted order, and metadata blocks of 2 KB per
    // (128 features, 128 k).  Otherwise the packed weight: kept values and index words.
    const void* w;
    const void* meta;
    const uint16_t* bias;
    int rows, out, in;
    int nt;            // token rows per pair tile
    uint8_t level;     // WsLevel
    uint8_t steps_per_warp;   // 16-column steps each epilogue warp of a quarter takes
    uint8_t act;       // epilogue activation (0 none, 1 GELU) on acc + bias
    int words_per_row; // of the index words
    int tiles_f;       // F
    int groups;        // G
    int row_tiles;     // ceil(rows / nt)
    uint32_t idesc;
};

constexpr int kGroupMax = 68;   // layers per launch (kernel parameters are limited to 32 KB)

template <int kMaxLayers>
struct alignas(64) WsGroup {
    WsLayer layer[kMaxLayers];
    int n_layers;
    int stages;
    int stage_bytes;   // one pipeline stage: kStageK / 64 quarters of (largest nt / 2) rows of 128 bytes
    uint32_t* dev_status;
    CUtensorMap map_r; // kEpiResidual: the residual, boxes as map_y's
};

// 128 k of a row of the packed weight: whole words of values and, but for half a word at 1:8, of index fields.
template <int M, int N>
struct PackedBlock {
    static constexpr int kCount = 16 / M * N, kBits = kCount * (M == 4 ? 2 : M == 8 ? 3 : 4);      // of a segment of 16 k
    static constexpr int kIdxBits = 8 * kBits, kIdxWords = kIdxBits % 32 ? 2 : kIdxBits / 32;
    uint4 v[kCount];
    uint32_t f[kIdxWords];

    __device__ __forceinline__ void load(const uint16_t* vals_row, const uint32_t* idx_row, int kb)
    {
        const uint4* src = reinterpret_cast<const uint4*>(vals_row) + kb * kCount;
#pragma unroll
        for (int i = 0; i < kCount; ++i) v[i] = __ldg(src + i);
        const int bit0 = kb * kIdxBits;
        // As wide as the words allow (rows are whole blocks of 128 k): a load of a warp touches 32 rows however little it takes of each
        // (2:4 word by word: 3152 x 1024 -> 4096 23.1 us, like this 21.2).
        if constexpr (kIdxWords == 4) {
            const uint4 t = __ldg(reinterpret_cast<const uint4*>(idx_row) + kb);
            f[0] = t.x; f[1] = t.y; f[2] = t.z; f[3] = t.w;
        } else if constexpr (kIdxBits == 64) {
            const uint2 t = __ldg(reinterpret_cast<const uint2*>(idx_row) + kb);
            f[0] = t.x; f[1] = t.y;
        } else {
#pragma unroll
            for (int i = 0; i < kIdxWords; ++i) f[i] = __ldg(idx_row + (bit0 >> 5) + i);
        }
        if constexpr (kIdxBits % 32 != 0) {      // 48 bits from bit 0 or 16 on
            f[0] = __funnelshift_r(f[0], f[1], bit0 & 31);
            f[1] >>= bit0 & 31;
        }
    }
    __device__ __forceinline__ uint32_t word(int i) const
    {
        const uint4& u = v[i >> 2];
        return (i & 3) == 0 ? u.x : (i & 3) == 1 ? u.y : (i & 3) == 2 ? u.z : u.w;
    }
    __device__ __forceinline__ Segment segment(int i) const
    {
        Segment s;
        s.v[0] = s.v[1] = s.v[2] = s.v[3] = 0u;
        if constexpr (kCount == 1) s.v[0] = word(i >> 1) >> (16 * (i & 1)) & 0xFFFFu;
#pragma unroll
        for (int j = 0; j < kCount / 2; ++j) s.v[j] = word(i * (kCount / 2) + j);
        const int bit = i * kBits, w0 = bit >> 5;
        s.fields = (bit & 31) + kBits > 32 ? __funnelshift_r(f[w0], f[w0 + 1 < kIdxWords ? w0 + 1 : w0], bit & 31) : f[w0] >> (bit & 31);
        return s;
    }
};

// A warp's blocks of 128 k, straight from the packed weight into tensor memory: 32 columns of values and 4 of metadata each.
// A lane expands its own feature's row; a metadata word holds 16 k of two rows eight apart (lane l: rows l % 8 and l % 8 + 8
// of its 16, the half of the 32 k that bit 3 of l says), so the nibbles change lanes by two shuffles a word.  All of a
// block's loads are in flight together (the next block's under them spill).
template <int M, int N>
__device__ __forceinline__ void write_packed(const uint16_t* vals_row, const uint32_t* idx_row, bool row_ok, int first, int blocks, int step,
                                             uint32_t a_col0, uint32_t e_col0)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int kb = first; kb < blocks; kb += step) {
        PackedBlock<M, N> cur;
        cur.load(vals_row, idx_row, kb);
        uint32_t e[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {          // 32 k
            uint32_t v[8], nib[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                uint4 t = sp24_words<M, N>(cur.segment(2 * h + i), nib[i]);
                if (!row_ok) {                 // a feature past the last one: zeros, four empty chunks of 4
                    t = make_uint4(0u, 0u, 0u, 0u);
                    nib[i] = 0x4444u;
                }
                v[4 * i] = t.x; v[4 * i + 1] = t.y; v[4 * i + 2] = t.z; v[4 * i + 3] = t.w;
            }
            tmem_st_32x32b_x8(a_col0 + (uint32_t)(32 * kb + 8 * h), v);
            const uint32_t mine = nib[0] | nib[1] << 16;
            const uint32_t lo = __shfl_sync(0xFFFFFFFFu, mine, lane & 23), hi = __shfl_sync(0xFFFFFFFFu, mine, (lane & 23) | 8);
            e[h] = prmt(lo, hi, lane & 8 ? 0x7632u : 0x5410u);
        }
        tmem_st_32x32b_x4(e_col0 + (uint32_t)(4 * kb), e);
    }
}

// A lane's row of the packed weight of a table's layer to come, the lines shared out among a quarter's warps, into L2: the activations leave
// no weight there from one call to the next, and the whole pair waits for a block that comes from HBM (an image has just been written).
// Four blocks of dim 256 at 64 images and 2:4, 119.4 us without it, 117.1 with it (and with images).
__device__ __forceinline__ void prefetch_packed(const WsLayer& L, int f, int part)
{
    const int row = f < L.out ? f : L.out - 1;
    const int pitch = L.in / kBlockK * (16 << (L.level & 1) << (2 - (L.level >> 1)));        // bytes of a row of values
    const uint8_t* vals = static_cast<const uint8_t*>(L.w) + (size_t)row * (size_t)pitch;
    for (int b = part * 128; b < pitch; b += kEpiParts * 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(vals + b));
    const uint32_t* idx = static_cast<const uint32_t*>(L.meta) + (size_t)row * (size_t)L.words_per_row;
    for (int i = part * 32; i < L.words_per_row; i += kEpiParts * 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(idx + i));
}

// kEpi: kEpiGelu, the instantiation whose epilogue applies the layer's activation, and kEpiResidual, which adds a residual, are for
// single-layer launches.  The residual comes by TMA into the staging buffer, in the rows that the result leaves by, while the tile is
// multiplied, and ldmatrix brings it to the lanes the way stmatrix takes the result back: as a pass of its own over four
// tensors it cost a LayerNorm 64 us where the plain one takes 34 (50432 rows of 768).
// kImage: the weight block comes from an image (masked form; with both ways in one instantiation the expansions' registers cost that
// form 1.3 us, 12608 x 768 -> 3072 at 1:8 37.1 -> 38.4).
template <bool kBf16, int kMaxLayers, int kEpi, bool kImage>
__global__ void __launch_bounds__(kThreads, 1)
linear_tc_sp24_ws_kernel(const __grid_constant__ WsGroup<kMaxLayers> p)
{
    constexpr bool kAct = kEpi == kEpiGelu, kRes = kEpi == kEpiResidual;
    constexpr bool kRuns = kAct || kMaxLayers > 1;      // how the rows leave, see the epilogue
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t cta_rank = cluster_ctarank();
    const int pair = blockIdx.x >> 1;

    const uint32_t staging_base = smem_base + (uint32_t)(p.stages * p.stage_bytes);
    const uint32_t bar_off = (uint32_t)(p.stages * p.stage_bytes) + kStagingTotal;
    const uint32_t bar_base = smem_base + bar_off;
    const uint32_t full_bar = bar_base;                       // leader only
    const uint32_t empty_bar = bar_base + 8 * kMaxStages;     // per CTA
    const uint32_t tmem_full_bar = bar_base + 16 * kMaxStages;        // per CTA
    const uint32_t tmem_empty_bar = tmem_full_bar + 8 * kNumAccum;    // leader only
    const uint32_t w_ready_bar = tmem_empty_bar + 8 * kNumAccum;      // leader only
    const uint32_t layer_bar = w_ready_bar + 8;                       // per CTA: epilogue warps between layers
    const uint32_t res_bar = layer_bar + 8;                           // kEpiResidual: one per epilogue warp
    const uint32_t holder_off = bar_off + 16 * kMaxStages + 16 * kNumAccum + 16 + 8 * kEpiWarps;
    volatile uint32_t* tmem_holder = reinterpret_cast<volatile uint32_t*>(smem_gen + holder_off);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem_gen + holder_off + 4);

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(full_bar + 8 * s, 1);
            mbar_init(empty_bar + 8 * s, 1);
        }
        for (int a = 0; a < kNumAccum; ++a) {
            mbar_init(tmem_full_bar + 8 * a, 1);
            mbar_init(tmem_empty_bar + 8 * a, 2 * kEpiWarps);
        }
        mbar_init(w_ready_bar, 2 * kEpiWarps);
        mbar_init(layer_bar, kEpiWarps);
        if constexpr (kRes)
            for (int w = 0; w < kEpiWarps; ++w) mbar_init(res_bar + 8 * w, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
    }
    if (warp == 1) tmem_alloc_pair(smem_base + holder_off, kTmemCols);
    tc_fence_before();
    __syncthreads();
    cluster_arrive();
    cluster_wait();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    pdl_wait_for_predecessors();
    pdl_release_successors();

    if (warp == 0) {
        // ------------------------------------------------ producer: this CTA's half of the activation rows
        // (whole warp converged, one elected lane issues: see the MMA warp).  One 3-D copy per stage
        // brings the four 64-wide K quarters of the stage: [quarter][row][128 bytes]; quarters beyond `in`
        // (a last stage of 128) arrive as zeros and are not multiplied.
        {
            const bool elected = elect_one();
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int li = 0; ok && li < p.n_layers; ++li) {
                const WsLayer& L = p.layer[li];
                if (pair >= L.groups * L.tiles_f) continue;
                const int half_rows = L.nt >> 1;
                const uint32_t tx_bytes = (uint32_t)(2 * (kStageK / 64) * half_rows * 128);   // both CTAs' boxes, in full
                const int num_k_stages = (L.in + kStageK - 1) / kStageK;
                for (int r = pair / L.tiles_f; ok && r < L.row_tiles; r += L.groups) {
                    const int r0 = r * L.nt + (int)cta_rank * half_rows;
                    for (int ks = 0; ks < num_k_stages; ++ks) {
                        ok = mbar_wait(empty_bar + 8 * stage, phase ^ 1u, abort_flag, p.dev_status, 1);
                        ok = __all_sync(0xFFFFFFFFu, ok);
                        if (!ok) break;
                        const uint32_t dst = smem_base + (uint32_t)(stage * p.stage_bytes);
                        const uint32_t bar = mapa_shared(full_bar + 8 * stage, 0);
                        if (elected) {
                            if (cta_rank == 0) mbar_arrive_expect_tx(full_bar + 8 * stage, tx_bytes);
                            tma_load_3d_pair(dst, &L.map_x, bar, 0, r0, (kStageK / 64) * ks);
                        }
                        __syncwarp();
                        if (++stage == p.stages) { stage = 0; phase ^= 1u; }
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer (leader CTA only)
        // The whole warp walks the loop and waits on the barriers; one elected lane issues, through a
        // predicate inside each instruction's asm block.  With the warp converged the descriptors stay in
        // uniform registers and no branch surrounds the instruction: measured ~36 cycles per MMA, against
        // ~80 with `if (elected)` around it and more with a single thread inside a divergent branch.
        if (cta_rank == 0) {
            const uint32_t elected = elect_one() ? 1u : 0u;
            // the base address was read from shared memory into an ordinary register; a warp reduction
            // returns it in a uniform one, so that every address derived from it stays uniform too
            const uint32_t tmem_u = __reduce_or_sync(0xFFFFFFFFu, tmem_base);
            int stage = 0;
            uint32_t phase = 0;
            int acc = 0;
            uint32_t acc_phase = 0;
            uint32_t w_phase = 0;
            bool ok = true;
            for (int li = 0; ok && li < p.n_layers; ++li) {
                const WsLayer& L = p.layer[li];
                if (pair >= L.groups * L.tiles_f) continue;
                const int g = pair / L.tiles_f;
                if (g >= L.row_tiles) continue;
                // the weight block of this layer is in tensor memory (both CTAs)
                ok = mbar_wait(w_ready_bar, w_phase, abort_flag, p.dev_status, 7);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                w_phase ^= 1u;
                tc_fence_after();
                const uint32_t a_col0 = tmem_u + (uint32_t)(kNumAccum * L.nt);
                const uint32_t e_col0 = a_col0 + (uint32_t)(L.in >> 2);
                const uint32_t idesc = L.idesc;
                const int num_k_stages = (L.in + kStageK - 1) / kStageK;
                const bool half_tail = (L.in % kStageK) != 0;      // the last stage holds 128 of K only
                const uint32_t quarter = (uint32_t)(L.nt * 64) >> 4;   // descriptor units between K quarters
                for (int r = g; ok && r < L.row_tiles; r += L.groups) {
                    ok = mbar_wait(tmem_empty_bar + 8 * acc, acc_phase ^ 1u, abort_flag, p.dev_status, 2);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_u + (uint32_t)(acc * L.nt);
                    for (int ks = 0; ks < num_k_stages; ++ks) {
                        ok = mbar_wait(full_bar + 8 * stage, phase, abort_flag, p.dev_status, 3);
                        ok = __all_sync(0xFFFFFFFFu, ok);
                        if (!ok) break;
                        tc_fence_after();
                        const uint64_t b_desc0 = smem_desc_k_major_sw128(smem_base + (uint32_t)(stage * p.stage_bytes));
                        const uint32_t a_col = a_col0 + (uint32_t)(ks * 8 * (kStageK / kSpUmmaK));
                        const uint32_t e_col = e_col0 + (uint32_t)(ks * (kStageK / kSpUmmaK));
                        // operands are computed by the whole warp (they stay uniform); only the instruction
                        // itself is predicated on the elected lane
                        if (half_tail && ks == num_k_stages - 1) {
#pragma unroll
                            for (int j = 0; j < kStageK / kSpUmmaK / 2; ++j) {
                                const uint64_t b_desc = b_desc0 + (uint64_t)((uint32_t)(j >> 1) * quarter + 4u * (uint32_t)(j & 1));
                                umma_sp_f16_pair_ts(d_tmem, a_col + (uint32_t)(8 * j), b_desc, e_col + (uint32_t)j, idesc,
                                                    (uint32_t)((ks | j) != 0), elected);
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < kStageK / kSpUmmaK; ++j) {
                                const uint64_t b_desc = b_desc0 + (uint64_t)((uint32_t)(j >> 1) * quarter + 4u * (uint32_t)(j & 1));
                                umma_sp_f16_pair_ts(d_tmem, a_col + (uint32_t)(8 * j), b_desc, e_col + (uint32_t)j, idesc,
                                                    (uint32_t)((ks | j) != 0), elected);
                            }
                        }
                        umma_commit_pair_if(empty_bar + 8 * stage, 3, elected);
                        if (++stage == p.stages) { stage = 0; phase ^= 1u; }
                    }
                    if (!ok) break;
                    umma_commit_pair_if(tmem_full_bar + 8 * acc, 3, elected);
                    if (++acc == kNumAccum) { acc = 0; acc_phase ^= 1u; }
                }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ weight loader + epilogue: lanes are features
        const int q = warp & 3;                 // TMEM lane quarter this warp may touch
        const int part = (warp - 2) >> 2;       // which of the quarter's warps
        const uint32_t empty_remote = mapa_shared(tmem_empty_bar, 0);
        const uint32_t w_ready_remote = mapa_shared(w_ready_bar, 0);
        const uint32_t lane_base = tmem_base + ((uint32_t)(q * 32) << 16);
        int acc = 0;
        uint32_t acc_phase = 0;
        uint32_t layer_phase = 0;
        uint32_t res_phase = 0;
        (void)res_phase;
        const uint32_t buf = staging_base + (uint32_t)((warp - 2) * kStagingBytes);
        // Lane t holds feature 8 * (t % 4) + t / 4 of the quarter's 32.  The staging buffer is rows of 32
        // features (64 bytes, no swizzle); one stmatrix.x4.trans writes 8 token rows: lane t gives the
        // address of (row 2 * (t / 8) + (t & 1), features 8 * ((t % 8) / 2) ...), and the two rows of a
        // matrix are 128 consecutive bytes, so no two of its addresses share a bank.
        const int feat_in_quarter = 8 * (lane & 3) + (lane >> 2);
        const uint32_t st_addr = buf + (uint32_t)((2 * (lane >> 3) + (lane & 1)) * 64 + ((lane & 7) >> 1) * 16);

        bool ok = true;
        bool first_layer = true;
        for (int li = 0; ok && li < p.n_layers; ++li) {
            const WsLayer& L = p.layer[li];
            if (pair >= L.groups * L.tiles_f) continue;
            const int g = pair / L.tiles_f;
            if (g >= L.row_tiles) continue;
            const int ft128 = (pair % L.tiles_f) * 2 + (int)cta_rank;
            const int f0 = ft128 * kFeatPerCta + q * 32;
            const int f = f0 + feat_in_quarter;
            const int l_rows = L.rows, l_out = L.out, nt = L.nt;
            const bool f_ok = f < l_out;

            // The column ranges of accumulators and weight block depend on the layer, and the warps of a
            // quarter read different columns of the same lanes: nobody writes the new weight block before
            // every epilogue warp of this CTA has read its last accumulator of the previous layer.
            if (!first_layer) {
                __syncwarp();
                if (lane == 0) mbar_arrive(layer_bar);
                ok = mbar_wait(layer_bar, layer_phase, abort_flag, p.dev_status, 8);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                layer_phase ^= 1u;
            }
            first_layer = false;

            // ---- this warp's share of the weight block into tensor memory.  Every MMA of the previous
            // layer has completed: this warp waited for the accumulator of that layer's last tile.  Image
            // row (block base + TMEM lane) is already the row of the feature this lane holds.
            {
                const uint32_t a_col0 = lane_base + (uint32_t)(kNumAccum * nt);
                const uint32_t e_col0 = a_col0 + (uint32_t)(L.in >> 2);
                if constexpr (kImage) {
                    const int a_chunks = L.in >> 6;          // 16 columns (64 bytes) each
                    const uint4* a_row = static_cast<const uint4*>(L.w) + (size_t)(ft128 * kFeatPerCta + q * 32 + lane) * (size_t)(L.in >> 4);
                    const bool blk_ok = ft128 * kFeatPerCta < l_out;     // rows of a started block of 32 exist (zero beyond out)
                    const bool row_ok = f0 < l_out;
                    for (int c = part; c < a_chunks; c += kEpiParts) {
                        uint32_t v[16];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            uint4 t = make_uint4(0u, 0u, 0u, 0u);
                            if (row_ok) t = __ldg(a_row + 4 * c + i);
                            v[4 * i] = t.x; v[4 * i + 1] = t.y; v[4 * i + 2] = t.z; v[4 * i + 3] = t.w;
                        }
                        tmem_st_32x32b_x16(a_col0 + (uint32_t)(16 * c), v);
                    }
                    const uint4* e_blk = static_cast<const uint4*>(L.meta) +
                                         (size_t)(blk_ok ? ft128 : 0) * (size_t)(L.in / kBlockK) * 128 + (size_t)(q * 32 + lane);
                    for (int kb = part; kb < L.in / kBlockK; kb += kEpiParts) {
                        uint4 t = make_uint4(0u, 0u, 0u, 0u);
                        if (blk_ok) t = __ldg(e_blk + (size_t)kb * 128);
                        uint32_t v[4] = {t.x, t.y, t.z, t.w};
                        tmem_st_32x32b_x4(e_col0 + (uint32_t)(4 * kb), v);
                    }
                } else {
                    const int row = f_ok ? f : l_out - 1;      // always one that can be read
                    const uint16_t* vals = static_cast<const uint16_t*>(L.w);
                    const uint32_t* idx_row = static_cast<const uint32_t*>(L.meta) + (size_t)row * (size_t)L.words_per_row;
                    auto block = [&](auto m, auto n) {
                        constexpr int M = decltype(m)::value, N = decltype(n)::value;
                        write_packed<M, N>(vals + (size_t)row * (size_t)(L.in / M * N), idx_row, f_ok, part, L.in / kBlockK, kEpiParts, a_col0, e_col0);
                    };
                    using std::integral_constant;
                    switch (L.level) {
                    case LEVEL_1_4: block(integral_constant<int, 4>{}, integral_constant<int, 1>{}); break;
                    case LEVEL_2_4: block(integral_constant<int, 4>{}, integral_constant<int, 2>{}); break;
                    case LEVEL_1_8: block(integral_constant<int, 8>{}, integral_constant<int, 1>{}); break;
                    case LEVEL_2_8: block(integral_constant<int, 8>{}, integral_constant<int, 2>{}); break;
                    case LEVEL_1_16: block(integral_constant<int, 16>{}, integral_constant<int, 1>{}); break;
                    default: block(integral_constant<int, 16>{}, integral_constant<int, 2>{}); break;
                    }
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster_release(w_ready_remote);
            }
            if constexpr (kMaxLayers > 1) {
                for (int next = li + 1; next < p.n_layers; ++next) {
                    const WsLayer& A = p.layer[next];
                    if (pair >= A.groups * A.tiles_f || pair / A.tiles_f >= A.row_tiles) continue;
                    prefetch_packed(A, ((pair % A.tiles_f) * 2 + (int)cta_rank) * kFeatPerCta + q * 32 + feat_in_quarter, part);
                    break;
                }
            }
            const float bias_f = (L.bias != nullptr && f_ok) ? bias_to_float<kBf16>(__ldg(L.bias + f)) : 0.f;
            const uint64_t bias2 = f32x2(bias_f, bias_f);
            const int l_act = kAct ? L.act : 0;
            (void)l_act;
            // this warp's run of token columns: steps of 16, [first_step, first_step + my_steps)
            const int total_steps = nt / kStepCols;
            const int first_step = part * L.steps_per_warp;
            int my_steps = total_steps - first_step;
            if (my_steps > L.steps_per_warp) my_steps = L.steps_per_warp;
            if (my_steps < 0) my_steps = 0;

            for (int r = g; r < L.row_tiles; r += L.groups) {
                const int row0 = r * nt + first_step * kStepCols;
                const bool has_res = kRes && f0 < l_out && my_steps > 0 && row0 < l_rows;
                (void)has_res;
                if constexpr (kRes) {
                    if (has_res && lane == 0) {
                        bulk_wait_group_read<0>();          // the stores of the previous tile have drained the buffer
                        const int last = l_rows - row0 < my_steps * kStepCols ? (l_rows - row0 + kStepCols - 1) / kStepCols : my_steps;
                        mbar_arrive_expect_tx(res_bar + 8 * (warp - 2), (uint32_t)(last * kStepCols * 64));
                        for (int s = 0; s < last; ++s)
                            tma_load_2d(buf + (uint32_t)(s * kStepCols * 64), &p.map_r, res_bar + 8 * (warp - 2), f0, row0 + s * kStepCols);
                    }
                    __syncwarp();
                }
                ok = mbar_wait(tmem_full_bar + 8 * acc, acc_phase, abort_flag, p.dev_status, 4);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after();
                const uint32_t t_col = lane_base + (uint32_t)(acc * nt + first_step * kStepCols);
                // all of this warp's columns are requested at once and the accumulator goes back to the MMA
                // warp before anything is converted
                uint32_t rr[kMaxSteps][16];
#pragma unroll
                for (int s = 0; s < kMaxSteps; ++s)
                    if (s < my_steps) tmem_ld_32x32b_x16(t_col + (uint32_t)(s * kStepCols), rr[s]);
                if (my_steps > 0) tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive_cluster(empty_remote + 8 * acc);
                    bulk_wait_group_read<0>();   // the stores of the previous tile have drained the buffer
                }
                __syncwarp();
                if constexpr (kRes) {
                    if (has_res) {
                        ok = mbar_wait(res_bar + 8 * (warp - 2), res_phase, abort_flag, p.dev_status, 9);
                        ok = __all_sync(0xFFFFFFFFu, ok);
                        if (!ok) break;
                        res_phase ^= 1u;
                    }
                }
#pragma unroll
                for (int s = 0; s < kMaxSteps; ++s) {
                    if (s >= my_steps) continue;
                    uint32_t w[8];
                    if constexpr (kRes) {
                        // (of a step past the last row, or features past the last one, what the buffer held; nothing of it is stored)
                        ldmatrix_x4_trans(st_addr + (uint32_t)(s * kStepCols * 64), w[0], w[1], w[2], w[3]);
                        ldmatrix_x4_trans(st_addr + (uint32_t)(s * kStepCols * 64 + 512), w[4], w[5], w[6], w[7]);
#pragma unroll
                        for (int j = 0; j < 8; ++j) w[j] = finish_pair_residual<kBf16>(rr[s][2 * j], rr[s][2 * j + 1], bias2, w[j]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            w[j] = finish_pair<kBf16, kAct>(rr[s][2 * j], rr[s][2 * j + 1], bias2, l_act);
                    }
                    stmatrix_x4_trans(st_addr + (uint32_t)(s * kStepCols * 64), w[0], w[1], w[2], w[3]);
                    stmatrix_x4_trans(st_addr + (uint32_t)(s * kStepCols * 64 + 512), w[4], w[5], w[6], w[7]);
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (f0 < l_out) {
                        // With GELU the warps are short of issue slots and a run leaves as one store (50432 x 768 -> 3072 138
                        // -> 131 us), and so it does in tables, whose layers follow one another without a gap (a DeiT-B block
                        // of 12608 rows 129.3 us, 130.5 by steps); a layer on its own as one store a step, which start while the
                        // rest is on its way: 65536 x 768 -> 3072 136 us, 144 by runs, back to back 141.2 and 142.2.
                        if (kRuns && my_steps == L.steps_per_warp) {
                            if (row0 < l_rows) tma_store_2d(&L.map_run, buf, f0, row0);
                        } else {
#pragma unroll
                            for (int s = 0; s < kMaxSteps; ++s)
                                if (s < my_steps && row0 + s * kStepCols < l_rows)
                                    tma_store_2d(&L.map_y, buf + (uint32_t)(s * kStepCols * 64), f0, row0 + s * kStepCols);
                        }
                    }
                    bulk_commit_group();
                }
                if (++acc == kNumAccum) { acc = 0; acc_phase ^= 1u; }
            }
        }
        if (lane == 0) bulk_wait_group_all();
        __syncwarp();
    }

    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(10000);
    }
    cluster_arrive();
    cluster_wait();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

// Token rows per pair tile for a layer of this input width: the largest multiple of 16, at most
// kMaxRowTile, such that two accumulators fit beside the weight block and its metadata; 0 if none does.
int ws_row_tile(int in)
{
    const int left = kTmemCols - in / 4 - in / 32;
    int nt = left / kNumAccum / kStepCols * kStepCols;
    if (nt > kMaxRowTile) nt = kMaxRowTile;
    return nt >= 64 ? nt : 0;
}

// Row tile of a layer whose rows `groups` row groups share: the busiest group takes its tiles one after the other, each in a time
// that goes with its rows and a fixed share, so narrower tiles pay where the widest leave a group's last one to few of the groups.
// Us with the widest and with the choice: 5319 x 512 -> 1536 at 2:8 11.5, 11.1; 3940 x 384 -> 1152 at 1:8 8.4, 8.1; 9000 x 768 -> 768
// at 1:8 10.5, 10.3; 3152 x 768 -> 2304 and larger launches the same.
int ws_layer_row_tile(int in, int rows, int groups)
{
    const int most = ws_row_tile(in);
    int best = most;
    long long best_cost = -1;
    for (int nt = most; nt >= 64; nt -= kStepCols) {
        const long long tiles = (rows + nt - 1) / nt;
        const long long cost = (tiles + groups - 1) / groups * (nt + 32);
        if (best_cost < 0 || cost < best_cost) { best = nt; best_cost = cost; }
    }
    return best;
}

template <bool kBf16, int kMaxLayers, int kEpi, bool kImage = false>
elsa_status launch_ws_group(const SparseJob* jobs, int n, elsa_dtype dtype, uint32_t* dev_status, cudaStream_t stream,
                            const DeviceInfo& dev)
{
    constexpr bool kRuns = kEpi == kEpiGelu || kMaxLayers > 1;
    auto kernel = linear_tc_sp24_ws_kernel<kBf16, kMaxLayers, kEpi, kImage>;
    const int fixed = kStagingTotal + kBarrierBytes + 1024;
    int max_nt = 0;
    for (int i = 0; i < n; ++i) {
        const int nt = ws_row_tile(jobs[i].in);
        if (nt > max_nt) max_nt = nt;
    }
    if (max_nt == 0) return fail(ELSA_ERR_SHAPE, "in=%d does not fit the weight-stationary sparse kernel", jobs[0].in);
    // a stage slot is sized for the widest row tile of the launch, so that narrow tiles still keep
    // the same number of activation bytes in flight
    const int stage_bytes = (kStageK / 64) * (max_nt / 2) * 128;
    int stages = (int)((dev.smem_optin - fixed) / stage_bytes);
    if (stages > kMaxStages) stages = kMaxStages;
    if (stages < 2) return fail(ELSA_ERR_CUDA, "not enough shared memory for two pipeline stages");
    const size_t smem = (size_t)stages * stage_bytes + fixed;

    static std::atomic<int> max_pairs[64];   // zero-initialised; racing first calls compute the same value
    const int slot = dev.device & 63;
    if (max_pairs[slot].load(std::memory_order_acquire) == 0) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dev.smem_optin) !=
            cudaSuccess) {
            cudaError_t e = cudaGetLastError();
            return fail(ELSA_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
        }
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)dev.sm_count);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = dev.smem_optin;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int m = 0;
        if (cudaOccupancyMaxActiveClusters(&m, kernel, &cfg) != cudaSuccess || m < 1) {
            cudaError_t e = cudaGetLastError();
            return fail(ELSA_ERR_CUDA, "cudaOccupancyMaxActiveClusters: %s", cudaGetErrorString(e));
        }
        max_pairs[slot].store(m, std::memory_order_release);
    }
    const int pairs = max_pairs[slot].load(std::memory_order_acquire);

    static WsGroup<kMaxLayers> g;   // host staging of the kernel parameters
    static std::mutex g_mutex;
    std::lock_guard<std::mutex> lock(g_mutex);
    const uint32_t fmt = dtype == ELSA_BF16 ? 1u : 0u;
    int used_pairs = 0;
    for (int i = 0; i < n; ++i) {
        const SparseJob& j = jobs[i];
        WsLayer& L = g.layer[i];
        L.tiles_f = (j.out + kPairFeat - 1) / kPairFeat;
        if (ws_row_tile(j.in) == 0 || j.in % kBlockK != 0 || L.tiles_f > pairs)
            return fail(ELSA_ERR_SHAPE, "in=%d out=%d does not fit the weight-stationary sparse kernel", j.in, j.out);
        L.nt = ws_layer_row_tile(j.in, j.rows, pairs / L.tiles_f);
        L.rows = j.rows; L.out = j.out; L.in = j.in;
        L.steps_per_warp = (uint8_t)((L.nt / kStepCols + kEpiParts - 1) / kEpiParts);
        L.row_tiles = (j.rows + L.nt - 1) / L.nt;
        L.groups = pairs / L.tiles_f;
        if (L.groups > L.row_tiles) L.groups = L.row_tiles;
        if (L.groups * L.tiles_f > used_pairs) used_pairs = L.groups * L.tiles_f;
        L.bias = j.bias;
        L.act = (uint8_t)j.act;
        if constexpr (!kImage) {
            L.w = j.w;
            L.meta = j.idx;
            L.level = j.M == 4 ? (j.N == 1 ? LEVEL_1_4 : LEVEL_2_4) : j.M == 8 ? (j.N == 1 ? LEVEL_1_8 : LEVEL_2_8) : j.N == 1 ? LEVEL_1_16 : LEVEL_2_16;
            L.words_per_row = (int)index_words_per_row(j.in, j.N, j.M);
        } else {
            L.w = j.workspace;
            L.meta = (const uint8_t*)j.workspace + sp24_meta_offset(j.out, j.in);
            L.level = 0;
            L.words_per_row = 0;
        }
        // sparse flag, fp32 accumulate, A and B of type fmt, K-major, N = nt, M = 256 over the pair
        L.idesc = (1u << 2) | (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(L.nt >> 3) << 17) |
                  ((uint32_t)(kPairFeat >> 4) << 24);
        elsa_status st;
        if ((st = make_map_x_quarters(&L.map_x, j.X, (uint64_t)j.in, (uint64_t)j.rows, (uint32_t)(L.nt / 2), kStageK / 64)) != ELSA_OK) return st;
        if ((st = make_map_2d(&L.map_y, j.Y, (uint64_t)j.out, (uint64_t)j.rows, 32, kStepCols, CU_TENSOR_MAP_SWIZZLE_NONE,
                              "Y")) != ELSA_OK)
            return st;
        if (kRuns && (st = make_map_2d(&L.map_run, j.Y, (uint64_t)j.out, (uint64_t)j.rows, 32, (uint32_t)(kStepCols * L.steps_per_warp),
                                       CU_TENSOR_MAP_SWIZZLE_NONE, "Y")) != ELSA_OK)
            return st;
    }
    if (kEpi == kEpiResidual) {
        const elsa_status st = make_map_2d(&g.map_r, jobs[0].residual, (uint64_t)jobs[0].out, (uint64_t)jobs[0].rows, 32, kStepCols,
                                           CU_TENSOR_MAP_SWIZZLE_NONE, "the residual");
        if (st != ELSA_OK) return st;
    }
    g.n_layers = n;
    g.stages = stages;
    g.stage_bytes = stage_bytes;
    g.dev_status = dev_status;

    ProfileScope scope(ELSA_KERNEL_LINEAR_TC_SP24_WS, stream);
    cudaError_t e = launch_pdl(kernel, dim3((unsigned)(2 * used_pairs)), dim3(kThreads), smem, stream, 2, g);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(ELSA_ERR_CUDA, "launch of linear_tc_sp24_ws failed: %s", cudaGetErrorString(e));
    }
    return launched("linear_tc_sp24_ws");
}

}  // namespace

int linear_tc_sparse_ws_group_max() { return kGroupMax; }

bool linear_tc_sparse_ws_suits(int in, int out, int N, int sm_count)
{
    return linear_tc_sparse_suits(in, N) && in % kBlockK == 0 && in <= kMaxIn && ws_row_tile(in) != 0 &&
           (out + kPairFeat - 1) / kPairFeat <= sm_count / 2;
}

elsa_status launch_linear_tc_sparse_ws_group(const SparseJob* jobs, int n, elsa_dtype dtype, uint32_t* dev_status,
                                             cudaStream_t stream)
{
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    if (n < 1 || n > kGroupMax) return fail(ELSA_ERR_SHAPE, "a grouped launch carries 1 to %d layers, got %d", kGroupMax, n);
    bool alone = false, image = false;
    for (int i = 0; i < n; ++i) {
        alone = alone || jobs[i].act != 0 || jobs[i].residual != nullptr;
        image = image || jobs[i].w == nullptr;
    }
    if (image) {
        if (n > 1 || alone) return fail(ELSA_ERR_SHAPE, "an image of the weight in a table or a chain of this kernel");
        return dtype == ELSA_BF16 ? launch_ws_group<true, 1, kEpiPlain, true>(jobs, 1, dtype, dev_status, stream, dev)
                                  : launch_ws_group<false, 1, kEpiPlain, true>(jobs, 1, dtype, dev_status, stream, dev);
    }
    if (alone) {
        // layers with an activation or a residual in the epilogue run one per launch, on the instantiation that has it
        for (int i = 0; i < n; ++i) {
            if (jobs[i].act != 0 && jobs[i].residual != nullptr) return fail(ELSA_ERR_SHAPE, "an activation and a residual in one epilogue of this kernel");
            if (jobs[i].residual != nullptr)
                st = dtype == ELSA_BF16 ? launch_ws_group<true, 1, kEpiResidual>(jobs + i, 1, dtype, dev_status, stream, dev)
                                        : launch_ws_group<false, 1, kEpiResidual>(jobs + i, 1, dtype, dev_status, stream, dev);
            else
                st = dtype == ELSA_BF16 ? launch_ws_group<true, 1, kEpiGelu>(jobs + i, 1, dtype, dev_status, stream, dev)
                                        : launch_ws_group<false, 1, kEpiGelu>(jobs + i, 1, dtype, dev_status, stream, dev);
            if (st != ELSA_OK) return st;
        }
        return ELSA_OK;
    }
    if (n == 1)
        return dtype == ELSA_BF16 ? launch_ws_group<true, 1, kEpiPlain>(jobs, 1, dtype, dev_status, stream, dev)
                                  : launch_ws_group<false, 1, kEpiPlain>(jobs, 1, dtype, dev_status, stream, dev);
    return dtype == ELSA_BF16 ? launch_ws_group<true, kGroupMax, kEpiPlain>(jobs, n, dtype, dev_status, stream, dev)
                              : launch_ws_group<false, kGroupMax, kEpiPlain>(jobs, n, dtype, dev_status, stream, dev);
}

}  // namespace elsa

// Multi-head self-attention of the ViT block between the pruned qkv and proj linears (ELSA, Sec. 3: the paper
// prunes the four linear modules and leaves the attention products dense; Sec. 4.2 measures whole models).
//     a[img, :, h] = softmax(q k^T / sqrt d) v      per image and head, over the keys of the same image
// with q, k, v the head's 64 columns in the three thirds of qkv [images * tokens][3 * dim].
//
// Work item = (128 query rows, head, image); tokens <= 256, head dimension 64 (the ViT / DeiT shapes) or 32 (Swin).
// An "image" is whatever set of consecutive rows attends within itself: for Swin, one window of the rolled grid, with
// an additive fp32 table per head on the scores (relative-position bias) and a second one per window position
// (the seam mask of shifted windows); the biased form is an instantiation of its own.  Both
// products run on tcgen05 with everything between them kept on chip:
//   1. TMA brings the Q tile, all K rows and all V rows of the head into shared memory (128-byte swizzle; a 3-D
//      tensor map [image][token][column] zero-fills the rows past the image's last token).
//   2. S = Q K^T: four MMAs (K = 16 each) into Tk = tokens rounded up to 16 fp32 columns of tensor memory.
//   3. Four warps, one query row per lane: p = 2^(s * log2(e) / 8 - ref) with ref at or just below the row's maximum
//      (see `rise`), row sum in fp32, p rounded to the 16-bit type and written back into tensor memory as the A
//      operand of the second product, two keys per column, over the low half of the columns S occupied.
//   4. O = P V: Tk / 16 MMAs with A from tensor memory and V as it lies in memory (keys outermost: MN-major
//      descriptor) into 64 columns of the part of S that is dead by then.
//   5. The same four warps read O, divide by the row sum, round once and store it, whole rows at a time.
// Persistent: one CTA per SM walks the items with the stride of the grid, with several items in flight: two for up
// to 256 keys, four for up to 128 (Swin's windows), each with its own shared-memory stage (Q, K, V), its own share
// of tensor memory (256 or 128 columns) and its own group of four softmax warps: item n uses stage, share and group
// n % 2 (n % 4).  The producer warp loads ahead as stages come free (Q and K of a stage after the scores of its
// previous item, V after that item's second product); the MMA warp issues S of item n, then P V of the
// oldest item whose probabilities are due, so one group's softmax runs under the others' products and epilogues.
// Every wait is bounded as in the GEMM kernels.
// What bounds it is an item's chain on its four warps (256 images x 12 heads of 197 tokens, cycles of the 6700 an item takes
// with another in flight): exponentials 4200 (11 a score for a warp alone, where the special-function unit asks for 8),
// second product 900 to 1300, output 900, the rest barriers.  113 -> 78 us against a maximum pass of its own (1400), tests
// for padded keys on every score, a row of the output per lane (1300 to 2200) and the item's divisions on the chain.
// Two warps to a quarter, half the keys each, with or without the two items exponentiating by turns: 89 and 107 us; units
// of 64 scores: 103.
#include <atomic>
#include <mutex>
#include <type_traits>

#include "elsa_attention_common.cuh"

namespace elsa {
namespace {

constexpr int kMaxHeadDim = 64;
constexpr int kQRows = 128;          // query rows per item = TMEM lanes
constexpr int kMaxTokens = 256;
constexpr int kTmemCols = 512;
constexpr int kGroupWarps = 4;       // softmax warps per group, one per TMEM lane quarter
constexpr int kQBytes = kQRows * kMaxHeadDim * 2;          // the shared-memory slots are laid out for head dimension 64

// kBufs items in flight per CTA: 2 for up to 256 keys (256 tensor-memory columns each), 4 for up to 128 keys (the
// windows of Swin), where an item's on-chip chain is short and only more of them in flight fill the SM.
template <int kD, int kBufs, bool kBias>
struct Shape {
    static constexpr int kBufCols = kTmemCols / kBufs;
    static constexpr int kThreads = (2 + kBufs * kGroupWarps) * 32;
    static constexpr int kKvBytes = (kBufs == 2 ? 256 : 128) * kMaxHeadDim * 2;
    static constexpr int kStageBytes = kQBytes + 2 * kKvBytes;
    static constexpr int kOutCols = kBufs == 2 ? kMaxHeadDim : 32;     // output columns a softmax warp stages at a time
    static constexpr int kOutBytes = 32 * kOutCols * 2;
    static constexpr int kSmemBytes = kBufs * (kStageBytes + kGroupWarps * kOutBytes) + 1024 /* alignment */ + 512 /* barriers */;
    static constexpr int kBiasUnit = kBufs == 2 ? 32 : 16;  // score columns a softmax warp handles at a time (registers):
    static constexpr int kUnit = kBufs == 4 && kD == 32 && !kBias ? 16 : 32;   // adding the tables; exponentiating
};

struct AttnParams {
    CUtensorMap map_q;    // box 64 columns x 128 tokens x 1 image
    CUtensorMap map_kv;   // box 64 columns x Tk tokens x 1 image
    uint16_t* out;        // [images * tokens][dim]
    int tokens, tk, dim;
    int m_tiles, heads, items;   // items = images * heads * m_tiles, query tile fastest
    int o_col;            // first column of O inside an item's half of tensor memory
    uint32_t idesc_s, idesc_o;
    uint32_t* dev_status;
    // biased form: scores get bias[head][row][key] + mask[image % n_masks][row][key] (fp32, rows of bias_pitch floats)
    const float* bias;
    const float* mask;    // or NULL
    int n_masks, bias_pitch;
};

// MN-major tile of rows of 64 bytes (32 16-bit values along N per reduction index) with the 64-byte swizzle: 8
// reduction rows form a 512-byte group.
__device__ __forceinline__ uint64_t smem_desc_mn_major_sw64(uint32_t addr, uint32_t block_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((block_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}

// D[tmem] (+)= A[tmem] * B[smem]: A's 16-bit values two per column, lane = row.  Predicated as the other forms.
__device__ __forceinline__ void umma_f16_ts_if(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate, uint32_t issue)
{
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "setp.ne.b32 q, %5, 0;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
        "}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(issue)
        : "memory");
}

__device__ __forceinline__ void tmem_ld_32x32b_x8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

template <bool kBf16, int kD, bool kBias, int kBufs>
__global__ void __launch_bounds__(Shape<kD, kBufs, kBias>::kThreads, 1) attention_kernel(const __grid_constant__ AttnParams p)
{
    static_assert(kD == 64 || kD == 32, "head dimension");
    static_assert(kBufs == 2 || kBufs == 4, "items in flight");
    constexpr int kBufCols = Shape<kD, kBufs, kBias>::kBufCols, kStageBytes = Shape<kD, kBufs, kBias>::kStageBytes, kKvBytesMax = Shape<kD, kBufs, kBias>::kKvBytes;
    constexpr int U = Shape<kD, kBufs, kBias>::kUnit, B = Shape<kD, kBufs, kBias>::kBiasUnit;
    constexpr int kLag = kBufs - 1;                   // P V of item n - kLag is issued after S of item n
    constexpr int kHeadDim = kD;
    constexpr int kItemQBytes = kQRows * kD * 2;      // bytes TMA delivers for the Q tile; K and V: tk * kD * 2
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t out_base = smem_base + kBufs * kStageBytes;
    const uint32_t bars = out_base + kBufs * kGroupWarps * Shape<kD, kBufs, kBias>::kOutBytes;
    // per buffer b: +0 qk_full, +8 v_full, +16 qk_empty, +24 s_full, +32 p_full, +40 o_full, +48 tmem_empty, +56 v_empty
    auto bar = [&](int which, int b) { return bars + (uint32_t)(64 * b + 8 * which); };
    enum { kQkFull = 0, kVFull, kQkEmpty, kSFull, kPFull, kOFull, kTmemEmpty, kVEmpty };
    const uint32_t tmem_holder_addr = bars + 64 * kBufs;
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem_raw + (tmem_holder_addr - smem_u32(smem_raw)));
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem_raw + (bars + 64 * kBufs + 8 - smem_u32(smem_raw)));

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int first = blockIdx.x, stride = gridDim.x;
    const int n_items = first < p.items ? (p.items - first + stride - 1) / stride : 0;   // items of this CTA

    if (warp == 1) {
        if (lane == 0) {
            for (int b = 0; b < kBufs; ++b) {
                mbar_init(bar(kQkFull, b), 1);
                mbar_init(bar(kVFull, b), 1);
                mbar_init(bar(kQkEmpty, b), 1);
                mbar_init(bar(kVEmpty, b), 1);
                mbar_init(bar(kSFull, b), 1);
                mbar_init(bar(kPFull, b), kGroupWarps);
                mbar_init(bar(kOFull, b), 1);
                mbar_init(bar(kTmemEmpty, b), kGroupWarps);
            }
            *abort_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        tmem_alloc(tmem_holder_addr, kTmemCols);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    pdl_wait_for_predecessors();
    pdl_release_successors();

    bool ok = true;
    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        const bool elected = elect_one();
        // Q and K of a stage are free as soon as the scores of its previous item are complete, V only after that item's
        // second product.  The loop asks for Q and K of item n, then for V of item n - 1: the order in which the MMA
        // warp frees them (S of item n - kBufs, then P V of item n - 1 - kBufs), so the next item's Q and K arrive under
        // the softmax, off the chain of the buffer, and no wait holds back a load whose stage is free already.
        for (int n = 0; ok && n <= n_items; ++n) {
            if (n < n_items) {
                const int b = n % kBufs;
                const uint32_t ph = (uint32_t)((n / kBufs) & 1);
                ok = mbar_wait(bar(kQkEmpty, b), ph ^ 1u, abort_flag, p.dev_status, 20);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                const int item = first + n * stride;
                const int mt = item % p.m_tiles, head = (item / p.m_tiles) % p.heads, img = item / (p.m_tiles * p.heads);
                const uint32_t q_smem = smem_base + (uint32_t)(b * kStageBytes);
                if (elected) {
                    mbar_arrive_expect_tx(bar(kQkFull, b), (uint32_t)(kItemQBytes + p.tk * kHeadDim * 2));
                    tma_load_3d(q_smem, &p.map_q, bar(kQkFull, b), head * kHeadDim, mt * kQRows, img);
                    tma_load_3d(q_smem + kQBytes, &p.map_kv, bar(kQkFull, b), p.dim + head * kHeadDim, 0, img);
                }
                __syncwarp();
            }
            if (n >= 1) {
                const int m = n - 1, b = m % kBufs;
                const uint32_t ph = (uint32_t)((m / kBufs) & 1);
                ok = mbar_wait(bar(kVEmpty, b), ph ^ 1u, abort_flag, p.dev_status, 27);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                const int item = first + m * stride;
                const int head = (item / p.m_tiles) % p.heads, img = item / (p.m_tiles * p.heads);
                const uint32_t q_smem = smem_base + (uint32_t)(b * kStageBytes);
                if (elected) {
                    mbar_arrive_expect_tx(bar(kVFull, b), (uint32_t)(p.tk * kHeadDim * 2));
                    tma_load_3d(q_smem + kQBytes + kKvBytesMax, &p.map_kv, bar(kVFull, b), 2 * p.dim + head * kHeadDim, 0, img);
                }
                __syncwarp();
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer: S of item n, then P V of item n - 1
        const uint32_t elected = elect_one() ? 1u : 0u;
        const uint32_t tmem_u = __reduce_or_sync(0xFFFFFFFFu, tmem_base);
        const int steps = p.tk / 16;
        for (int n = 0; ok && n < n_items + kLag; ++n) {
            if (n < n_items) {
                const int b = n % kBufs;
                const uint32_t ph = (uint32_t)((n / kBufs) & 1);
                ok = mbar_wait(bar(kTmemEmpty, b), ph ^ 1u, abort_flag, p.dev_status, 21);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                ok = mbar_wait(bar(kQkFull, b), ph, abort_flag, p.dev_status, 22);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after();
                const uint32_t q_smem = smem_base + (uint32_t)(b * kStageBytes);
                const uint64_t a_desc = kD == 64 ? smem_desc_k_major_sw128(q_smem) : smem_desc_k_major_sw64(q_smem);
                const uint64_t b_desc = kD == 64 ? smem_desc_k_major_sw128(q_smem + kQBytes) : smem_desc_k_major_sw64(q_smem + kQBytes);
#pragma unroll
                for (int k = 0; k < kHeadDim / 16; ++k)
                    umma_f16_if(tmem_u + (uint32_t)(b * kBufCols), a_desc + (uint64_t)(2 * k), b_desc + (uint64_t)(2 * k), p.idesc_s,
                                (uint32_t)(k != 0), elected);
                umma_commit_if(bar(kSFull, b), elected);
                umma_commit_if(bar(kQkEmpty, b), elected);     // Q and K of the stage have been read
            }
            if (n >= kLag) {
                const int m = n - kLag, b = m % kBufs;
                const uint32_t ph = (uint32_t)((m / kBufs) & 1);
                ok = mbar_wait(bar(kVFull, b), ph, abort_flag, p.dev_status, 23);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                ok = mbar_wait(bar(kPFull, b), ph, abort_flag, p.dev_status, 24);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after();
                const uint32_t t_buf = tmem_u + (uint32_t)(b * kBufCols);
                const uint32_t v_smem = smem_base + (uint32_t)(b * kStageBytes + kQBytes + kKvBytesMax);
                const uint64_t v_desc = kD == 64 ? smem_desc_mn_major_sw128(v_smem, (uint32_t)(p.tk * kHeadDim * 2))
                                                 : smem_desc_mn_major_sw64(v_smem, (uint32_t)(p.tk * kHeadDim * 2));
                // 16 keys of kD * 2 bytes per MMA
                for (int k = 0; k < steps; ++k)
                    umma_f16_ts_if(t_buf + (uint32_t)p.o_col, t_buf + (uint32_t)(8 * k), v_desc + (uint64_t)(k * (16 * kD * 2 >> 4)),
                                   p.idesc_o, (uint32_t)(k != 0), elected);
                umma_commit_if(bar(kOFull, b), elected);
                umma_commit_if(bar(kVEmpty, b), elected);      // V of the stage has been read
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ softmax and output: group g takes the items n = g, g + 2, ...
        const int g = (warp - 2) / kGroupWarps;
        const int quarter = warp & 3;                                  // the TMEM lanes this warp may touch
        const uint32_t stage_out = out_base + (uint32_t)((warp - 2) * Shape<kD, kBufs, kBias>::kOutBytes);
        constexpr float kFar = 32768.f;     // no probability above it: inside the 16-bit types and far inside fp32
        const float scale = (kD == 64 ? 0.125f : 0.17677669529663687f) * 1.4426950408889634f;   // log2(e) / sqrt(kD)
        int mt, head, img, next_mt = 0, next_head = 0, next_img = 0;
        auto decode = [&](int n) {
            const int item = first + n * stride;
            next_mt = item % p.m_tiles; next_head = (item / p.m_tiles) % p.heads; next_img = item / (p.m_tiles * p.heads);
        };
        decode(g);
        for (int n = g; ok && n < n_items; n += kBufs) {
            const uint32_t ph = (uint32_t)((n / kBufs) & 1);
            mt = next_mt; head = next_head; img = next_img;
            const int row = mt * kQRows + quarter * 32 + lane;         // token index inside the image
            const uint32_t t_lane = tmem_base + (uint32_t)(g * kBufCols) + ((uint32_t)(quarter * 32) << 16);
            if (mt * kQRows + quarter * 32 >= p.tokens) {
                // none of its rows exists: the warp only keeps its place in the barriers
                ok = mbar_wait(bar(kSFull, g), ph, abort_flag, p.dev_status, 25);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                if (lane == 0) mbar_arrive(bar(kPFull, g));
                if (n + kBufs < n_items) decode(n + kBufs);
                ok = mbar_wait(bar(kOFull, g), ph, abort_flag, p.dev_status, 26);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                if (lane == 0) mbar_arrive(bar(kTmemEmpty, g));
                continue;
            }
            float sum = 0.f;
            // biased form: what is exponentiated is s * scale + (bias + mask) * log2(e); the tables' rows of this lane
            const float* brow = nullptr;
            const float* mrow = nullptr;
            if constexpr (kBias) {
                if (row < p.tokens) {
                    brow = p.bias + ((size_t)head * p.tokens + row) * (size_t)p.bias_pitch;
                    if (p.mask != nullptr) mrow = p.mask + ((size_t)(img % p.n_masks) * p.tokens + row) * (size_t)p.bias_pitch;
                }
            }
            // (bias + mask) * log2(e) for `count` columns from col0 (multiples of 4; rows of the tables are 16-byte
            // aligned and padded to bias_pitch, so whole float4 loads stay inside a row); zeros without tables
            auto load_bias = [&](float* bb, int col0, int count) {
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    if (4 * v >= count) break;
                    float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (brow != nullptr && col0 + 4 * v < p.bias_pitch) {
                        b4 = __ldg(reinterpret_cast<const float4*>(brow + col0) + v);
                        if (mrow != nullptr) {
                            const float4 m4 = __ldg(reinterpret_cast<const float4*>(mrow + col0) + v);
                            b4.x += m4.x; b4.y += m4.y; b4.z += m4.z; b4.w += m4.w;
                        }
                    }
                    bb[4 * v] = b4.x * 1.4426950408889634f; bb[4 * v + 1] = b4.y * 1.4426950408889634f;
                    bb[4 * v + 2] = b4.z * 1.4426950408889634f; bb[4 * v + 3] = b4.w * 1.4426950408889634f;
                }
            };
            // The bias table's values of one unit, as loaded (no arithmetic on them here, so a request stays in flight
            // until the values are used): the first unit is asked for before the scores are waited for, every other
            // one while the unit before it is worked on, which takes most of the L2 latency out of the item's chain.
            // The mask (shifted windows only) is read where it is used: a second array across the wait would spill.
            constexpr int kReq = kBias ? Shape<kD, kBufs, kBias>::kBiasUnit : 1;
            float bq[kReq];
            auto request = [&](int col0) {
#pragma unroll
                for (int v = 0; v < kReq / 4; ++v) {
                    float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (brow != nullptr && col0 + 4 * v < p.bias_pitch) b4 = __ldg(reinterpret_cast<const float4*>(brow + col0) + v);
                    bq[4 * v] = b4.x; bq[4 * v + 1] = b4.y; bq[4 * v + 2] = b4.z; bq[4 * v + 3] = b4.w;
                }
            };
            if constexpr (kBias) request(0);
            ok = mbar_wait(bar(kSFull, g), ph, abort_flag, p.dev_status, 25);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            {
                float m = -INFINITY;
                if constexpr (kBias) {
                    auto ld_unit = [&](uint32_t taddr, uint32_t (&r)[B]) {
                        if constexpr (B == 32) tmem_ld_32x32b_x32(taddr, r);
                        else tmem_ld_32x32b_x16(taddr, r);
                    };
                    const int units = p.tk / B;                      // whole units
                    const bool tail = B == 32 && (p.tk & 31) != 0;   // plus one chunk of 16
                    // first pass of the biased form: t = s * scale + (bias + mask) * log2(e) replaces s in tensor memory,
                    // so the tables are read once
                    for (int u = 0; u < units; ++u) {
                        uint32_t r[B];
                        float bb[B];
                        ld_unit(t_lane + (uint32_t)(B * u), r);
#pragma unroll
                        for (int v = 0; v < B / 4; ++v) {
                            float4 m4 = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (mrow != nullptr && B * u + 4 * v < p.bias_pitch) m4 = __ldg(reinterpret_cast<const float4*>(mrow + B * u) + v);
                            bb[4 * v] = (bq[4 * v] + m4.x) * 1.4426950408889634f;
                            bb[4 * v + 1] = (bq[4 * v + 1] + m4.y) * 1.4426950408889634f;
                            bb[4 * v + 2] = (bq[4 * v + 2] + m4.z) * 1.4426950408889634f;
                            bb[4 * v + 3] = (bq[4 * v + 3] + m4.w) * 1.4426950408889634f;
                        }
                        if (u + 1 < units) request(B * (u + 1));
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < B; ++j) {
                            const float t = fmaf(__uint_as_float(r[j]), scale, bb[j]);
                            r[j] = __float_as_uint(t);
                            if (B * u + j < p.tokens) m = fmaxf(m, t);
                        }
#pragma unroll
                        for (int h = 0; h < B / 16; ++h) {
                            uint32_t part[16];
#pragma unroll
                            for (int j = 0; j < 16; ++j) part[j] = r[16 * h + j];
                            tmem_st_32x32b_x16(t_lane + (uint32_t)(B * u + 16 * h), part);
                        }
                    }
                    if (tail) {
                        uint32_t r[16];
                        float bb[16];
                        tmem_ld_32x32b_x16(t_lane + (uint32_t)(B * units), r);
                        load_bias(bb, B * units, 16);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const float t = fmaf(__uint_as_float(r[j]), scale, bb[j]);
                            r[j] = __float_as_uint(t);
                            if (B * units + j < p.tokens) m = fmaxf(m, t);
                        }
                        tmem_st_32x32b_x16(t_lane + (uint32_t)(B * units), r);
                    }
                    tmem_wait_st();
                }
                // p = 2^(s * scale - ref) for 16 columns from col0, two scores an instruction where there is such an
                // instruction; eight packed pairs.  Only a unit with padded keys tests every column (at half rate).
                float ref = m;                                     // biased form: the row's maximum, in the exponent's domain already
                const uint64_t scale2 = f32x2(scale, scale);
                uint64_t sum2 = f32x2(0.f, 0.f);
                auto exp16 = [&](auto masked, const uint32_t* r, int col0, uint64_t& part2, uint32_t (&w)[8]) {
                    const uint64_t minus_ref = f32x2(-ref, -ref);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const uint64_t s2 = f32x2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
                        const float2 a = f32x2_split(kBias ? f32x2_add(s2, minus_ref) : f32x2_fma(s2, scale2, minus_ref));
                        float e0, e1;
                        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(a.x));
                        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(a.y));
                        if constexpr (decltype(masked)::value) {          // padded keys take no part
                            if (col0 + 2 * j >= p.tokens) e0 = 0.f;
                            if (col0 + 2 * j + 1 >= p.tokens) e1 = 0.f;
                        }
                        part2 = f32x2_add(part2, f32x2(e0, e1));
                        w[j] = pack2<kBf16>(e0, e1);
                    }
                };
                // Unbiased form: the reference is a whole number, the largest of the row's first unit rounded down.  Where the
                // probabilities of a later unit sum to more than kFar, it becomes that unit's largest, the sum and the
                // P columns written so far are multiplied by the power of two between the two (exact but for values
                // below the 16-bit type's normal range) and the unit is done again.  So no probability leaves the
                // 16-bit types' range, none is smaller than with the maximum of the row as the reference, and the
                // scores are read once: a pass for the maximum ahead of this one took a sixth of an item's time, a
                // maximum of each unit ahead of its exponentials as much (half-rate instructions in a serial chain).
                auto top_of = [&](auto masked, const uint32_t* r, int col0) {
                    float t0 = -INFINITY, t1 = -INFINITY;
#pragma unroll
                    for (int j = 0; j < U; j += 2) {
                        if (!decltype(masked)::value || col0 + j < p.tokens) t0 = fmaxf(t0, __uint_as_float(r[j]));
                        if (!decltype(masked)::value || col0 + j + 1 < p.tokens) t1 = fmaxf(t1, __uint_as_float(r[j + 1]));
                    }
                    return fmaxf(floorf(fmaxf(t0, t1) * scale), -3.0e38f);      // finite for scores of minus infinity
                };
                auto rise = [&](float to, int written) {
                    const float up = fminf(to - ref, 127.f);
                    const float factor = __uint_as_float((uint32_t)(127 - (int)up) << 23);         // 2^-up, 0 from 127 on
                    ref = to;
                    sum2 = f32x2_mul(sum2, f32x2(factor, factor));
                    tmem_wait_st();
                    for (int c = 0; c < written; c += 8) {
                        uint32_t w[8];
                        tmem_ld_32x32b_x8(t_lane + (uint32_t)c, w);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float2 v = raw2_to_float2<kBf16>(w[j]);
                            w[j] = pack2<kBf16>(v.x * factor, v.y * factor);
                        }
                        tmem_st_32x32b_x8(t_lane + (uint32_t)c, w);
                    }
                };
                // unit u, the first 16 columns of it where that is all there is (`halved`); P's columns lie over S columns of
                // units that have been read already.  A whole unit is one straight run of code: a warp has little else to
                // overlap its latencies with.
                auto columns = [&](auto masked, const uint32_t* r, int u, bool halved) {
                    uint64_t part2;
                    auto once = [&]() {
                        part2 = f32x2(0.f, 0.f);
#pragma unroll
                        for (int h = 0; h < U / 16; ++h) {
                            if (decltype(masked)::value && h == 1 && halved) break;
                            uint32_t w[8];
                            exp16(masked, r + 16 * h, U * u + 16 * h, part2, w);
                            tmem_st_32x32b_x8(t_lane + (uint32_t)(U / 2 * u + 8 * h), w);
                        }
                    };
                    once();
                    if constexpr (!kBias) {
                        const float2 part = f32x2_split(part2);
                        const bool far = part.x + part.y > kFar;
                        if (__any_sync(0xFFFFFFFFu, far)) {
                            const float top = top_of(masked, r, U * u);
                            rise(far && top > ref ? top : ref, U / 2 * u);
                            once();
                        }
                    }
                    sum2 = f32x2_add(sum2, part2);
                };
                auto unit = [&](const uint32_t* r, int u) {
                    if (U * u + U <= p.tokens) columns(std::false_type{}, r, u, false);
                    else columns(std::true_type{}, r, u, U * u + U > p.tk);
                };
                auto first_top = [&](const uint32_t* r) {
                    return U <= p.tokens ? top_of(std::false_type{}, r, 0) : top_of(std::true_type{}, r, 0);
                };
                // the last unit's load may reach past tk, inside the item's share of columns
                const int units = (p.tk + U - 1) / U;
                if constexpr (kBufs == 2) {
                    // the next unit's scores are on their way while one is exponentiated
                    uint32_t ra[U], rb[U];
                    tmem_ld_32x32b_x32(t_lane, ra);
                    if constexpr (!kBias) {
                        tmem_wait_ld();
                        ref = first_top(ra);
                    }
                    for (int u = 0; u < units; u += 2) {
                        tmem_wait_ld();
                        if (u + 1 < units) tmem_ld_32x32b_x32(t_lane + (uint32_t)(U * (u + 1)), rb);
                        unit(ra, u);
                        if (u + 1 < units) {
                            tmem_wait_ld();
                            if (u + 2 < units) tmem_ld_32x32b_x32(t_lane + (uint32_t)(U * (u + 2)), ra);
                            unit(rb, u + 1);
                        }
                    }
                } else {
                    // four groups of warps have each other's work to run under a load
                    for (int u = 0; u < units; ++u) {
                        uint32_t r[U];
                        if constexpr (U == 32) tmem_ld_32x32b_x32(t_lane + (uint32_t)(U * u), r);
                        else tmem_ld_32x32b_x16(t_lane + (uint32_t)(U * u), r);
                        tmem_wait_ld();
                        if (!kBias && u == 0) ref = first_top(r);
                        unit(r, u);
                    }
                }
                const float2 both = f32x2_split(sum2);
                sum = both.x + both.y;
            }
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kPFull, g));
            if (n + kBufs < n_items) decode(n + kBufs);                // its divisions run under the second product
            ok = mbar_wait(bar(kOFull, g), ph, abort_flag, p.dev_status, 26);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            const float inv = 1.0f / sum;
            // A lane has a row of the output; the rows leave through shared memory (16-byte vectors, swizzled), so that a
            // store instruction covers whole 64- or 128-byte rows instead of 16 bytes of 32 lines.
            constexpr int kCols = Shape<kD, kBufs, kBias>::kOutCols < kD ? Shape<kD, kBufs, kBias>::kOutCols : kD;
            constexpr int kVecs = kCols / 8, kRowsPerStore = 32 / kVecs;
#pragma unroll
            for (int c = 0; c < kD / kCols; ++c) {
                uint32_t o[kCols / 16][16];
#pragma unroll
                for (int q = 0; q < kCols / 16; ++q) tmem_ld_32x32b_x16(t_lane + (uint32_t)(p.o_col + kCols * c + 16 * q), o[q]);
                tmem_wait_ld();
                if (c == kD / kCols - 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kTmemEmpty, g));    // the share may take the S of item n + kBufs
                }
                const int sw = (kVecs == 8 ? lane : lane >> 1) & (kVecs - 1);
#pragma unroll
                for (int v = 0; v < kVecs; ++v) {
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        w[e] = pack2<kBf16>(__uint_as_float(o[v >> 1][8 * (v & 1) + 2 * e]) * inv, __uint_as_float(o[v >> 1][8 * (v & 1) + 2 * e + 1]) * inv);
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stage_out + (uint32_t)((lane * kVecs + (v ^ sw)) * 16)),
                                 "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                                 : "memory");
                }
                __syncwarp();
                const int row0 = mt * kQRows + quarter * 32;
                uint16_t* dst = p.out + ((size_t)img * p.tokens + row0) * (size_t)p.dim + head * kHeadDim + kCols * c;
                uint4 w[kVecs];
#pragma unroll
                for (int i = 0; i < kVecs; ++i) {
                    const int r = i * kRowsPerStore + lane / kVecs, v = lane & (kVecs - 1);
                    const int rsw = (kVecs == 8 ? r : r >> 1) & (kVecs - 1);
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[i].x), "=r"(w[i].y), "=r"(w[i].z), "=r"(w[i].w)
                                 : "r"(stage_out + (uint32_t)((r * kVecs + (v ^ rsw)) * 16)) : "memory");
                }
                uint16_t* at = dst + (size_t)(lane / kVecs) * (size_t)p.dim + 8 * (lane & (kVecs - 1));
#pragma unroll
                for (int i = 0; i < kVecs; ++i) {
                    if (row0 + i * kRowsPerStore + lane / kVecs < p.tokens) *reinterpret_cast<uint4*>(at) = w[i];
                    at += kRowsPerStore * p.dim;
                }
                __syncwarp();                                          // the staging rows have been read
            }
        }
    }
    if (!ok) let_copies_land();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

template <bool kBf16, int kD, bool kBias, int kBufs>
elsa_status launch(const AttnParams& p, int images, int heads, cudaStream_t stream, const DeviceInfo& dev)
{
    constexpr int kSmemBytes = Shape<kD, kBufs, kBias>::kSmemBytes, kThreads = Shape<kD, kBufs, kBias>::kThreads;
    auto kernel = attention_kernel<kBf16, kD, kBias, kBufs>;
    static std::atomic<bool> attr_set[64];
    const int slot = dev.device & 63;
    if (!attr_set[slot].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess) {
            cudaError_t e = cudaGetLastError();
            return fail(ELSA_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
        }
        attr_set[slot].store(true, std::memory_order_release);
    }
    (void)images;
    (void)heads;
    const dim3 grid((unsigned)(p.items < dev.sm_count ? p.items : dev.sm_count));   // one persistent CTA per SM
    ProfileScope scope(ELSA_KERNEL_ATTENTION, stream);
    cudaError_t e = launch_pdl(kernel, grid, dim3(kThreads), (size_t)kSmemBytes, stream, 1, p);
    if (e != cudaSuccess) return fail(ELSA_ERR_CUDA, "attention launch: %s", cudaGetErrorString(e));
    return launched("attention");
}

}  // namespace

bool attention_suits(int tokens, int heads, int dim)
{
    return tokens >= 1 && tokens <= kMaxTokens && heads >= 1 && (dim == heads * 64 || dim == heads * 32);
}

elsa_status launch_attention(const uint16_t* qkv, int images, int tokens, int heads, int dim, elsa_dtype dtype,
                             uint16_t* out, uint32_t* dev_status, cudaStream_t stream, const float* bias, const float* mask,
                             int n_masks, int bias_pitch)
{
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    if (!attention_suits(tokens, heads, dim))
        return fail(ELSA_ERR_SHAPE, "attention needs 1..%d tokens per image and a head dimension of 32 or 64 (tokens=%d, heads=%d, dim=%d)",
                    kMaxTokens, tokens, heads, dim);
    const int head_dim = dim / heads;
    if (bias == nullptr && mask != nullptr) return fail(ELSA_ERR_NULL, "a mask table needs a bias table");
    if (bias != nullptr && (bias_pitch < tokens || bias_pitch % 4 != 0 || (mask != nullptr && n_masks < 1)))
        return fail(ELSA_ERR_SHAPE, "bias_pitch=%d must be a multiple of 4 and at least tokens=%d, n_masks=%d at least 1", bias_pitch,
                    tokens, n_masks);
    if (bias != nullptr && ((((uintptr_t)bias) & 15u) != 0 || (((uintptr_t)mask) & 15u) != 0))
        return fail(ELSA_ERR_ALIGN, "the bias and mask tables must be 16-byte aligned");
    if ((long long)images * heads * ((tokens + kQRows - 1) / kQRows) > 0x7fffffffLL)
        return fail(ELSA_ERR_SHAPE, "images * heads does not fit an int");
    // windows that fit a warp's registers: 286 us here against 89 us there for 32768 windows x heads of 49 tokens
    if (window_attention_suits(tokens, heads, dim))
        return launch_window_attention(qkv, images, tokens, heads, dim, dtype, out, dev_status, stream, bias, mask, n_masks, bias_pitch, dev);
    // A call whose items leave SMs idle is bound by the chain of one: sixteen query rows a CTA instead of 128.
    if (bias == nullptr && attention_rows_suits(images, tokens, heads, head_dim, dev.sm_count))
        return launch_attention_rows(qkv, images, tokens, heads, dim, dtype, out, dev_status, stream, dev);
    AttnParams p;
    p.out = out;
    p.tokens = tokens;
    p.tk = (tokens + 15) / 16 * 16;
    p.dim = dim;
    p.m_tiles = (tokens + kQRows - 1) / kQRows;
    p.heads = heads;
    p.items = images * heads * p.m_tiles;
    // O (head_dim columns) over the part of S that P does not cover (P: tk / 2 columns from 0; S is dead by then)
    p.o_col = (p.tk / 2 + 31) / 32 * 32;
    const uint32_t fmt = dtype == ELSA_BF16 ? 1u : 0u;
    p.idesc_s = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(p.tk >> 3) << 17) | ((uint32_t)(kQRows >> 4) << 24);
    p.idesc_o = (1u << 4) | (fmt << 7) | (fmt << 10) | (1u << 16) | ((uint32_t)(head_dim >> 3) << 17) | ((uint32_t)(kQRows >> 4) << 24);
    p.dev_status = dev_status;
    p.bias = bias; p.mask = mask; p.n_masks = n_masks > 0 ? n_masks : 1; p.bias_pitch = bias_pitch;
    if ((st = make_map_qkv(&p.map_q, qkv, images, tokens, dim, head_dim, kQRows, "q")) != ELSA_OK) return st;
    if ((st = make_map_qkv(&p.map_kv, qkv, images, tokens, dim, head_dim, (uint32_t)p.tk, "k, v")) != ELSA_OK) return st;
    const bool bf = dtype == ELSA_BF16, biased = bias != nullptr;
    const bool four = p.tk <= 128;       // short chains: four items in flight per CTA
#define ELSA_ATTN(D, B, N) (bf ? launch<true, D, B, N>(p, images, heads, stream, dev) : launch<false, D, B, N>(p, images, heads, stream, dev))
    if (head_dim == 64) {
        if (biased) return four ? ELSA_ATTN(64, true, 4) : ELSA_ATTN(64, true, 2);
        return four ? ELSA_ATTN(64, false, 4) : ELSA_ATTN(64, false, 2);
    }
    if (biased) return four ? ELSA_ATTN(32, true, 4) : ELSA_ATTN(32, true, 2);
    return four ? ELSA_ATTN(32, false, 4) : ELSA_ATTN(32, false, 2);
#undef ELSA_ATTN
}

}  // namespace elsa

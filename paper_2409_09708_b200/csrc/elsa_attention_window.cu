// Window attention of the Swin block (heads of 32, at most 64 tokens per window) with the whole window in one warp:
//     a = softmax(q k^T / sqrt d + bias[head] + mask[window % n_masks]) v
//
// Why a kernel of its own beside elsa_attention.cu.  A 49-token window fills 49 of the 128 rows of a tcgen05 tile,
// and its chain  TMA -> S -> tensor-memory read -> softmax -> tensor-memory write -> P V -> tensor-memory read
// costs the same round trips as a full tile: that form was bound by the latency of the chain.  Here a warp keeps a
// window's K and V as mma.sync fragments in registers and walks its 16-row tiles: scores, softmax and probabilities
// never leave the registers (the accumulator of the first product is the A operand of the second), no barrier joins
// the warps, and twelve independent windows per SM hide each other's latencies.  mma.sync runs at 1024
// multiply-adds a cycle and SM, but the 120 instructions of a window are only 240 cycles; the special-function unit
// needs 224, and its q, k, v and a are 12.5 KB, 290 cycles of an SM's share of HBM.  Measured, 32768 windows x heads
// of 49 tokens (Swin-B's first stage at batch 128, 411 MB): 286 -> 89 us (4.6 TB/s), with a mask 341 -> 120 us; the
// 24 blocks of Swin-B 2738 -> 1037 us.
//
// A CTA belongs to one head, whose bias table it keeps in shared memory in the order of the accumulator fragments
// (scaled by log2 e; -inf at keys past the window's end, so nothing else masks them).  CTAs of different heads walk
// the same windows at the same time, so the 64-byte slices that the heads take from a row share L2 lines.
//
// Per warp: TMA brings q, k, v of the next window (3-D map [window][token][column]; rows past the window's last
// token are zero-filled) as soon as the current window's fragments are in registers; the result goes through
// shared memory and a TMA store, which clips at the window's last token.

#include <atomic>

#include "elsa_attention_common.cuh"

namespace elsa {
namespace {

constexpr int kWarps = 12;                 // 12 x 16 KB of tiles + 16 KB of bias fill shared memory; 168 registers each
constexpr int kThreads = kWarps * 32;
constexpr int kHeadDim = 32;
constexpr int kRows = 64;                  // rows of a tile in shared memory
constexpr int kTileBytes = kRows * kHeadDim * 2;
constexpr int kSlotBytes = 4 * kTileBytes; // q, k, v, a of one warp
constexpr int kRowTiles = kRows / 16;
constexpr int kMaxKeyTiles = 8;
constexpr int kBiasBytes = kRowTiles * kMaxKeyTiles * 32 * 16;
constexpr int kSmemBytes = kWarps * kSlotBytes + kBiasBytes + 256 /* barriers */ + 1024 /* alignment */;

struct WindowParams {
    CUtensorMap map_in;    // qkv, box 32 columns x 64 tokens x 1 window
    CUtensorMap map_out;   // a, same box
    const float* bias;     // [heads][tokens][pitch] or NULL
    const float* mask;     // [n_masks][tokens][pitch] (kMask)
    int windows, heads, tokens, pitch, n_masks, dim;
    int ctas_per_head;
    uint32_t* dev_status;
};

__device__ __forceinline__ void stmatrix_x4(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
                 : "memory");
}

__device__ __forceinline__ void tma_load_window(uint32_t dst, const CUtensorMap* map, uint32_t bar, int column, int window)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(column), "r"(0), "r"(window)
        : "memory");
}

__device__ __forceinline__ void tma_store_window(const CUtensorMap* map, uint32_t src, int column, int window)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(src), "r"(column), "r"(0), "r"(window)
                 : "memory");
}

// 16-byte unit `unit` of row `row` of a tile: rows of 64 bytes with TMA's 64-byte swizzle.
__device__ __forceinline__ uint32_t tile_addr(uint32_t tile, int row, int unit)
{
    return tile + (uint32_t)(row * 64) + (uint32_t)((unit ^ ((row >> 1) & 3)) << 4);
}

// kKeyTiles: 8-key column tiles of the scores, 7 for up to 56 keys (7 x 7 windows) and 8 for up to 64.  With a mask 6 for up to
// 48: there a window may end in any tile, in the other two forms in the last.  (Looking for the end in every tile cost 32768
// windows x heads of 49 tokens 122 us against 113.)
template <bool kBf16, bool kMask, int kKeyTiles>
__global__ void __launch_bounds__(kThreads, 1) window_attention_kernel(const __grid_constant__ WindowParams p)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;           // fragment row and column pair of this lane
    constexpr float kLog2e = 1.4426950408889634f;

    float4* bias_s = reinterpret_cast<float4*>(smem_gen + kWarps * kSlotBytes);
    const uint32_t bar = smem_base + kWarps * kSlotBytes + kBiasBytes + 8u * (uint32_t)warp;
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem_gen + kWarps * kSlotBytes + kBiasBytes + 8 * kWarps);
    const uint32_t tile_q = smem_base + (uint32_t)(warp * kSlotBytes);
    const uint32_t tile_k = tile_q + kTileBytes, tile_v = tile_q + 2 * kTileBytes, tile_o = tile_q + 3 * kTileBytes;

    if (lane == 0) mbar_init(bar, 1);
    if (threadIdx.x == 0) *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async_smem();
    __syncwarp();
    pdl_wait_for_predecessors();
    pdl_release_successors();

    const int head = (int)blockIdx.x % p.heads;
    const int step = p.ctas_per_head * kWarps;
    int window = (int)blockIdx.x / p.heads + p.ctas_per_head * warp;
    auto load = [&](int w) {
        if (lane == 0) {
            mbar_arrive_expect_tx(bar, 3 * kTileBytes);
            tma_load_window(tile_q, &p.map_in, bar, head * kHeadDim, w);
            tma_load_window(tile_k, &p.map_in, bar, p.dim + head * kHeadDim, w);
            tma_load_window(tile_v, &p.map_in, bar, 2 * p.dim + head * kHeadDim, w);
        }
    };
    if (window < p.windows) load(window);

    // the head's bias table in fragment order: entry (row tile, key tile, lane) holds the four scores of that lane
    for (int e = (int)threadIdx.x; e < kRowTiles * kKeyTiles * 32; e += kThreads) {
        const int el = e & 31, kt = (e >> 5) % kKeyTiles, rt = (e >> 5) / kKeyTiles;
        float v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int row = 16 * rt + (el >> 2) + 8 * (c >> 1), key = 8 * kt + 2 * (el & 3) + (c & 1);
            v[c] = key >= p.tokens ? -INFINITY
                   : (p.bias != nullptr && row < p.tokens) ? kLog2e * __ldg(p.bias + ((size_t)head * p.tokens + row) * p.pitch + key)
                                                           : 0.f;
        }
        bias_s[(rt * kMaxKeyTiles + kt) * 32 + el] = make_float4(v[0], v[1], v[2], v[3]);
    }
    __syncthreads();

    const float scale = 0.17677669529663687f * kLog2e;      // 1 / sqrt(32), in powers of two
    const int row_tiles = (p.tokens + 15) >> 4;
    // row and 16-byte unit that this lane addresses in the matrix loads and stores
    const int a_row = (lane & 7) + (lane & 8), a_unit = lane >> 4;   // rows 0-7, 8-15 of unit 0, then of unit 1
    uint32_t phase = 0;

    for (; window < p.windows; window += step) {
        bool ok = mbar_wait(bar, phase, abort_flag, p.dev_status, 31);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        phase ^= 1u;
        uint32_t kf[kKeyTiles][4];     // key tile: dims 0-7, 8-15, 16-23, 24-31
#pragma unroll
        for (int j = 0; j < kKeyTiles; ++j)
            ldmatrix_x4(tile_addr(tile_k, 8 * j + (lane & 7), lane >> 3), kf[j][0], kf[j][1], kf[j][2], kf[j][3]);
        uint32_t vf[4][8];             // 16 keys: (keys 0-7, keys 8-15) of dim tiles 0..3
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            ldmatrix_x4_trans(tile_addr(tile_v, 16 * s + a_row, a_unit), vf[s][0], vf[s][1], vf[s][2], vf[s][3]);
            ldmatrix_x4_trans(tile_addr(tile_v, 16 * s + a_row, 2 + a_unit), vf[s][4], vf[s][5], vf[s][6], vf[s][7]);
        }
        const float* mask_w = nullptr;
        if constexpr (kMask) mask_w = p.mask + (size_t)(window % p.n_masks) * p.tokens * p.pitch;

        // the previous window's result has left its tile
        if (lane == 0) bulk_wait_group_read<0>();
        __syncwarp();
#pragma unroll 1
        for (int rt = 0; rt < row_tiles; ++rt) {
            uint32_t qf[2][4];
            ldmatrix_x4(tile_addr(tile_q, 16 * rt + a_row, a_unit), qf[0][0], qf[0][1], qf[0][2], qf[0][3]);
            ldmatrix_x4(tile_addr(tile_q, 16 * rt + a_row, 2 + a_unit), qf[1][0], qf[1][1], qf[1][2], qf[1][3]);
            float s[kKeyTiles][4];
            float2 mk[kMask ? kKeyTiles : 1][2];
            if constexpr (kMask) {
                // rows past the window are discarded: any row's values do
                const int r0 = min(16 * rt + g, p.tokens - 1), r1 = min(16 * rt + g + 8, p.tokens - 1);
#pragma unroll
                for (int j = 0; j < kKeyTiles; ++j) {
                    const int key = 8 * j + 2 * t;
                    const bool in = key < p.tokens;
                    mk[j][0] = in ? __ldg(reinterpret_cast<const float2*>(mask_w + r0 * p.pitch + key)) : make_float2(0.f, 0.f);
                    mk[j][1] = in ? __ldg(reinterpret_cast<const float2*>(mask_w + r1 * p.pitch + key)) : make_float2(0.f, 0.f);
                    // the pair's second value may lie behind the window's last token: whatever is there, a NaN even, is nobody's
                    if ((kKeyTiles == 6 || j == kKeyTiles - 1) && key + 1 >= p.tokens) mk[j][0].y = mk[j][1].y = 0.f;
                }
            }
#pragma unroll
            for (int j = 0; j < kKeyTiles; ++j) {
                s[j][0] = s[j][1] = s[j][2] = s[j][3] = 0.f;
                mma_16816<kBf16>(s[j], qf[0], kf[j][0], kf[j][1]);
                mma_16816<kBf16>(s[j], qf[1], kf[j][2], kf[j][3]);
            }
            if (rt == row_tiles - 1) {
                // q, k and v are in registers: the slot takes the next window
                __syncwarp();
                if (window + step < p.windows) load(window + step);
            }
            float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
            for (int j = 0; j < kKeyTiles; ++j) {
                const float4 b = bias_s[(rt * kMaxKeyTiles + j) * 32 + lane];
                s[j][0] = fmaf(s[j][0], scale, b.x);
                s[j][1] = fmaf(s[j][1], scale, b.y);
                s[j][2] = fmaf(s[j][2], scale, b.z);
                s[j][3] = fmaf(s[j][3], scale, b.w);
                if constexpr (kMask) {
                    s[j][0] = fmaf(mk[j][0].x, kLog2e, s[j][0]);
                    s[j][1] = fmaf(mk[j][0].y, kLog2e, s[j][1]);
                    s[j][2] = fmaf(mk[j][1].x, kLog2e, s[j][2]);
                    s[j][3] = fmaf(mk[j][1].y, kLog2e, s[j][3]);
                }
                m0 = fmaxf(m0, fmaxf(s[j][0], s[j][1]));
                m1 = fmaxf(m1, fmaxf(s[j][2], s[j][3]));
            }
            m0 = fmaxf(m0, __shfl_xor_sync(0xFFFFFFFFu, m0, 1));
            m1 = fmaxf(m1, __shfl_xor_sync(0xFFFFFFFFu, m1, 1));
            m0 = fmaxf(m0, __shfl_xor_sync(0xFFFFFFFFu, m0, 2));
            m1 = fmaxf(m1, __shfl_xor_sync(0xFFFFFFFFu, m1, 2));
            float sum0 = 0.f, sum1 = 0.f;
            uint32_t pf[4][4];           // probabilities as A fragments of 16 keys each
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (j < kKeyTiles) {
                    const int jj = j < kKeyTiles ? j : 0;
                    const float e0 = exp2_approx(s[jj][0] - m0), e1 = exp2_approx(s[jj][1] - m0);
                    const float e2 = exp2_approx(s[jj][2] - m1), e3 = exp2_approx(s[jj][3] - m1);
                    sum0 += e0 + e1;
                    sum1 += e2 + e3;
                    pf[j >> 1][2 * (j & 1)] = pack2<kBf16>(e0, e1);
                    pf[j >> 1][2 * (j & 1) + 1] = pack2<kBf16>(e2, e3);
                } else {
                    pf[j >> 1][2 * (j & 1)] = 0u;
                    pf[j >> 1][2 * (j & 1) + 1] = 0u;
                }
            }
            float o[4][4];
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                o[d][0] = o[d][1] = o[d][2] = o[d][3] = 0.f;
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) mma_16816<kBf16>(o[d], pf[ks], vf[ks][2 * d], vf[ks][2 * d + 1]);
            }
            sum0 += __shfl_xor_sync(0xFFFFFFFFu, sum0, 1);
            sum1 += __shfl_xor_sync(0xFFFFFFFFu, sum1, 1);
            sum0 += __shfl_xor_sync(0xFFFFFFFFu, sum0, 2);
            sum1 += __shfl_xor_sync(0xFFFFFFFFu, sum1, 2);
            const float i0 = 1.0f / sum0, i1 = 1.0f / sum1;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                stmatrix_x4(tile_addr(tile_o, 16 * rt + a_row, 2 * h + a_unit),
                            pack2<kBf16>(o[2 * h][0] * i0, o[2 * h][1] * i0), pack2<kBf16>(o[2 * h][2] * i1, o[2 * h][3] * i1),
                            pack2<kBf16>(o[2 * h + 1][0] * i0, o[2 * h + 1][1] * i0),
                            pack2<kBf16>(o[2 * h + 1][2] * i1, o[2 * h + 1][3] * i1));
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
            tma_store_window(&p.map_out, tile_o, head * kHeadDim, window);
            bulk_commit_group();
        }
    }
    if (lane == 0) bulk_wait_group_all();
    __syncwarp();
    if (*abort_flag)
        // a wait gave up: let copies that may still be in flight land before shared memory is released
        for (int i = 0; i < 200; ++i) __nanosleep(10000);
}

elsa_status make_map_windows(CUtensorMap* map, const void* base, int windows, int tokens, int columns, const char* what)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return fail(ELSA_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    cuuint64_t dims[3] = {(cuuint64_t)columns, (cuuint64_t)tokens, (cuuint64_t)windows};
    cuuint64_t strides[2] = {(cuuint64_t)columns * 2, (cuuint64_t)tokens * (cuuint64_t)columns * 2};
    cuuint32_t box[3] = {kHeadDim, kRows, 1};
    cuuint32_t elem[3] = {1, 1, 1};
    CUresult rc = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT16, 3, const_cast<void*>(base), dims, strides, box, elem,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (rc != CUDA_SUCCESS) return fail(ELSA_ERR_CUDA, "tensor map for %s rejected (CUresult %d)", what, (int)rc);
    return ELSA_OK;
}

template <bool kBf16, bool kMask, int kKeyTiles>
elsa_status launch(const WindowParams& p, cudaStream_t stream, const DeviceInfo& dev)
{
    auto kernel = window_attention_kernel<kBf16, kMask, kKeyTiles>;
    static std::atomic<bool> attr_set[64];
    const int slot = dev.device & 63;
    if (!attr_set[slot].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess) {
            cudaError_t e = cudaGetLastError();
            return fail(ELSA_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
        }
        attr_set[slot].store(true, std::memory_order_release);
    }
    ProfileScope scope(ELSA_KERNEL_ATTENTION, stream);
    cudaError_t e = launch_pdl(kernel, dim3((unsigned)(p.heads * p.ctas_per_head)), dim3(kThreads), (size_t)kSmemBytes, stream, 1, p);
    if (e != cudaSuccess) return fail(ELSA_ERR_CUDA, "window attention launch: %s", cudaGetErrorString(e));
    return launched("window_attention");
}

}  // namespace

// Heads of 32 and at most 64 tokens: the whole window fits one warp's registers.
bool window_attention_suits(int tokens, int heads, int dim) { return tokens >= 1 && tokens <= kRows && dim == heads * kHeadDim; }

elsa_status launch_window_attention(const uint16_t* qkv, int windows, int tokens, int heads, int dim, elsa_dtype dtype, uint16_t* out,
                                    uint32_t* dev_status, cudaStream_t stream, const float* bias, const float* mask, int n_masks,
                                    int bias_pitch, const DeviceInfo& dev)
{
    WindowParams p;
    p.bias = bias; p.mask = mask;
    p.windows = windows; p.heads = heads; p.tokens = tokens; p.pitch = bias_pitch; p.n_masks = n_masks > 0 ? n_masks : 1; p.dim = dim;
    // one CTA per SM, an equal number per head (at least one; no more than its windows)
    p.ctas_per_head = dev.sm_count / heads;
    if (p.ctas_per_head > windows) p.ctas_per_head = windows;
    if (p.ctas_per_head < 1) p.ctas_per_head = 1;
    p.dev_status = dev_status;
    elsa_status st;
    if ((st = make_map_windows(&p.map_in, qkv, windows, tokens, 3 * dim, "qkv")) != ELSA_OK) return st;
    if ((st = make_map_windows(&p.map_out, out, windows, tokens, dim, "a")) != ELSA_OK) return st;
    const bool bf = dtype == ELSA_BF16;
#define ELSA_WATTN(MASK, TILES) (bf ? launch<true, MASK, TILES>(p, stream, dev) : launch<false, MASK, TILES>(p, stream, dev))
    if (mask == nullptr) return tokens <= 56 ? ELSA_WATTN(false, 7) : ELSA_WATTN(false, 8);
    return tokens <= 48 ? ELSA_WATTN(true, 6) : tokens <= 56 ? ELSA_WATTN(true, 7) : ELSA_WATTN(true, 8);
#undef ELSA_WATTN
}

}  // namespace elsa

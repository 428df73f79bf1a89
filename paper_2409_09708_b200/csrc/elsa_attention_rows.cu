// Multi-head self-attention without tables for calls of few images:
//     a[img, :, h] = softmax(q k^T / sqrt d) v
//
// Why a kernel of its own beside elsa_attention.cu.  There an item is 128 query rows of a head, one row a lane, and its chain
// (TMA, S, tensor-memory read, 208 exponentials a lane one after the other, tensor-memory write, P V, read, store) is 7000
// cycles; one image has 24 items for 148 SMs, so the call lasts as long as one chain.  Here a CTA has sixteen query rows of a
// head, 156 CTAs for that image, and its four warps share the keys: each multiplies its key tiles (mma.sync, scores and
// probabilities stay in registers, the accumulator of the first product is the A operand of the second), keeps its own
// maximum and sum, and the four parts are joined through shared memory.  K and V are read from L2 once for every sixteen rows,
// which is what makes this the slower form once the other one fills the SMs (see attention_rows_suits).
//
// TMA brings Q, K and V (rows past the image's last token are zero); padded keys are kept out by their scores.

#include <atomic>

#include "elsa_attention_common.cuh"

namespace elsa {
namespace {

constexpr int kWarps = 4;
constexpr int kThreads = kWarps * 32;
constexpr int kRows = 16;                      // query rows of a CTA
constexpr int kMostTiles = 256 / 16 / kWarps;  // key tiles of 16 a warp

struct RowsParams {
    CUtensorMap map_q;     // box kD columns x 16 tokens x 1 image
    CUtensorMap map_kv;    // box kD columns x tk tokens x 1 image
    uint16_t* out;         // [images * tokens][dim]
    int tokens, tk, dim, heads, row_tiles;
    uint32_t* dev_status;
};

// Floats of a warp's share of the output: rows a multiple of 8 banks apart but not of 32, so that the fragments' 8-byte stores
// fall on all banks.
template <int kD>
constexpr int kPitch = kD + 8;

template <int kD>
constexpr int rows_smem(int tk)
{
    return 1024 /* alignment */ + kRows * kD * 2 + 2 * tk * kD * 2 + kWarps * kRows * (kPitch<kD> + 2) * 4 + 32 /* barriers */;
}

// 16-byte unit `unit` of row `row` of a tile as TMA lays it out: rows of 128 or 64 bytes, swizzled over their width.
template <int kD>
__device__ __forceinline__ uint32_t unit_addr(uint32_t tile, int row, int unit)
{
    if constexpr (kD == 64) return tile + (uint32_t)(row * 128) + (uint32_t)((unit ^ (row & 7)) << 4);
    else return tile + (uint32_t)(row * 64) + (uint32_t)((unit ^ ((row >> 1) & 3)) << 4);
}

template <bool kBf16, int kD>
__global__ void __launch_bounds__(kThreads) attention_rows_kernel(const __grid_constant__ RowsParams p)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;           // fragment row and column pair of this lane
    const uint32_t tile_q = smem_base, tile_k = tile_q + kRows * kD * 2, tile_v = tile_k + (uint32_t)(p.tk * kD * 2);
    const int parts_off = kRows * kD * 2 + 2 * p.tk * kD * 2;
    float* parts = reinterpret_cast<float*>(smem_gen + parts_off);                  // [warp][row][kPitch]
    float* tops = parts + kWarps * kRows * kPitch<kD>;                              // [warp][row]
    float* sums = tops + kWarps * kRows;                                            // [warp][row]
    const int bar_off = parts_off + kWarps * kRows * (kPitch<kD> + 2) * 4;
    const uint32_t qk_bar = smem_base + (uint32_t)bar_off, v_bar = qk_bar + 8;
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem_gen + bar_off + 16);

    const int rt = (int)blockIdx.x % p.row_tiles, head = ((int)blockIdx.x / p.row_tiles) % p.heads, img = (int)blockIdx.x / (p.row_tiles * p.heads);
    if (threadIdx.x == 0) {
        mbar_init(qk_bar, 1);
        mbar_init(v_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
    }
    __syncthreads();
    pdl_wait_for_predecessors();
    pdl_release_successors();
    if (threadIdx.x == 0) {
        mbar_arrive_expect_tx(qk_bar, (uint32_t)((kRows + p.tk) * kD * 2));
        tma_load_3d(tile_q, &p.map_q, qk_bar, head * kD, rt * kRows, img);
        tma_load_3d(tile_k, &p.map_kv, qk_bar, p.dim + head * kD, 0, img);
        mbar_arrive_expect_tx(v_bar, (uint32_t)(p.tk * kD * 2));
        tma_load_3d(tile_v, &p.map_kv, v_bar, 2 * p.dim + head * kD, 0, img);
    }
    constexpr float kScale = (kD == 64 ? 0.125f : 0.17677669529663687f) * 1.4426950408889634f;   // log2(e) / sqrt(kD)
    float s[kMostTiles][2][4], o[kD / 8][4];
    float top0 = -INFINITY, top1 = -INFINITY, sum0 = 0.f, sum1 = 0.f;      // rows g and g + 8
#pragma unroll
    for (int n = 0; n < kD / 8; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;

    bool ok = mbar_wait(qk_bar, 0, abort_flag, p.dev_status, 60);
    if (!ok) let_copies_land();
    ok = __all_sync(0xFFFFFFFFu, ok);
    if (ok) {
        uint32_t q[kD / 16][4];
#pragma unroll
        for (int k = 0; k < kD / 16; ++k)
            ldmatrix_x4(unit_addr<kD>(tile_q, lane & 15, 2 * k + (lane >> 4)), q[k][0], q[k][1], q[k][2], q[k][3]);
#pragma unroll
        for (int i = 0; i < kMostTiles; ++i) {
            const int key0 = 16 * (warp + kWarps * i);
            if (key0 >= p.tk) break;
#pragma unroll
            for (int h = 0; h < 2; ++h) s[i][h][0] = s[i][h][1] = s[i][h][2] = s[i][h][3] = 0.f;
#pragma unroll
            for (int k = 0; k < kD / 16; ++k) {
                uint32_t b[4];
                ldmatrix_x4(unit_addr<kD>(tile_k, key0 + (lane & 7) + ((lane >> 4) << 3), 2 * k + ((lane >> 3) & 1)), b[0], b[1], b[2], b[3]);
                mma_16816<kBf16>(s[i][0], q[k], b[0], b[1]);
                mma_16816<kBf16>(s[i][1], q[k], b[2], b[3]);
            }
            if (key0 + 16 > p.tokens) {            // the last tile's padded keys take no part
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (key0 + 8 * h + 2 * t + (e & 1) >= p.tokens) s[i][h][e] = -INFINITY;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                top0 = fmaxf(top0, fmaxf(s[i][h][0], s[i][h][1]));
                top1 = fmaxf(top1, fmaxf(s[i][h][2], s[i][h][3]));
            }
        }
#pragma unroll
        for (int x = 1; x <= 2; x <<= 1) {
            top0 = fmaxf(top0, __shfl_xor_sync(0xFFFFFFFFu, top0, x));
            top1 = fmaxf(top1, __shfl_xor_sync(0xFFFFFFFFu, top1, x));
        }
        top0 = fmaxf(top0 * kScale, -3.0e38f);      // finite for scores of minus infinity, and for a warp without keys
        top1 = fmaxf(top1 * kScale, -3.0e38f);
        ok = mbar_wait(v_bar, 0, abort_flag, p.dev_status, 61);
        if (!ok) let_copies_land();
        ok = __all_sync(0xFFFFFFFFu, ok);
    }
    if (ok) {
#pragma unroll
        for (int i = 0; i < kMostTiles; ++i) {
            const int key0 = 16 * (warp + kWarps * i);
            if (key0 >= p.tk) break;
            uint32_t a[4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float e0 = exp2_approx(fmaf(s[i][h][0], kScale, -top0)), e1 = exp2_approx(fmaf(s[i][h][1], kScale, -top0));
                const float e2 = exp2_approx(fmaf(s[i][h][2], kScale, -top1)), e3 = exp2_approx(fmaf(s[i][h][3], kScale, -top1));
                sum0 += e0 + e1;
                sum1 += e2 + e3;
                a[2 * h] = pack2<kBf16>(e0, e1);
                a[2 * h + 1] = pack2<kBf16>(e2, e3);
            }
#pragma unroll
            for (int n = 0; n < kD / 8; n += 2) {
                uint32_t b[4];
                ldmatrix_x4_trans(unit_addr<kD>(tile_v, key0 + (lane & 15), n + (lane >> 4)), b[0], b[1], b[2], b[3]);
                mma_16816<kBf16>(o[n], a, b[0], b[1]);
                mma_16816<kBf16>(o[n + 1], a, b[2], b[3]);
            }
        }
#pragma unroll
        for (int x = 1; x <= 2; x <<= 1) {
            sum0 += __shfl_xor_sync(0xFFFFFFFFu, sum0, x);
            sum1 += __shfl_xor_sync(0xFFFFFFFFu, sum1, x);
        }
        float* mine = parts + (size_t)(warp * kRows + g) * kPitch<kD> + 2 * t;
#pragma unroll
        for (int n = 0; n < kD / 8; ++n) {
            *reinterpret_cast<float2*>(mine + 8 * n) = make_float2(o[n][0], o[n][1]);
            *reinterpret_cast<float2*>(mine + 8 * kPitch<kD> + 8 * n) = make_float2(o[n][2], o[n][3]);
        }
        if (t == 0) {
            tops[warp * kRows + g] = top0;
            tops[warp * kRows + g + 8] = top1;
            sums[warp * kRows + g] = sum0;
            sums[warp * kRows + g + 8] = sum1;
        }
    }
    __syncthreads();
    // one thread: eight columns of a row, the parts in the order of the warps
    constexpr int kUnits = kD / 8;
    const int r = (int)threadIdx.x / kUnits, unit = (int)threadIdx.x % kUnits;
    const int row = rt * kRows + r;
    if (ok && *abort_flag == 0 && r < kRows && row < p.tokens) {
        float top = tops[r];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) top = fmaxf(top, tops[w * kRows + r]);
        float sum = 0.f, v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float f = exp2_approx(tops[w * kRows + r] - top);
            sum = fmaf(sums[w * kRows + r], f, sum);
            const float4* src = reinterpret_cast<const float4*>(parts + (size_t)(w * kRows + r) * kPitch<kD> + 8 * unit);
            const float4 x = src[0], y = src[1];
            v[0] = fmaf(x.x, f, v[0]); v[1] = fmaf(x.y, f, v[1]); v[2] = fmaf(x.z, f, v[2]); v[3] = fmaf(x.w, f, v[3]);
            v[4] = fmaf(y.x, f, v[4]); v[5] = fmaf(y.y, f, v[5]); v[6] = fmaf(y.z, f, v[6]); v[7] = fmaf(y.w, f, v[7]);
        }
        const float inv = 1.0f / sum;
        *reinterpret_cast<uint4*>(p.out + ((size_t)img * p.tokens + row) * (size_t)p.dim + head * kD + 8 * unit) =
            make_uint4(pack2<kBf16>(v[0] * inv, v[1] * inv), pack2<kBf16>(v[2] * inv, v[3] * inv), pack2<kBf16>(v[4] * inv, v[5] * inv),
                       pack2<kBf16>(v[6] * inv, v[7] * inv));
    }
}

template <bool kBf16, int kD>
elsa_status launch(const RowsParams& p, int images, cudaStream_t stream, const DeviceInfo& dev)
{
    auto kernel = attention_rows_kernel<kBf16, kD>;
    static std::atomic<bool> attr_set[64];
    const int slot = dev.device & 63;
    if (!attr_set[slot].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, rows_smem<kD>(256)) != cudaSuccess) {
            cudaError_t e = cudaGetLastError();
            return fail(ELSA_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
        }
        attr_set[slot].store(true, std::memory_order_release);
    }
    ProfileScope scope(ELSA_KERNEL_ATTENTION, stream);
    cudaError_t e = launch_pdl(kernel, dim3((unsigned)(images * p.heads * p.row_tiles)), dim3(kThreads), (size_t)rows_smem<kD>(p.tk), stream, 1, p);
    if (e != cudaSuccess) return fail(ELSA_ERR_CUDA, "attention launch: %s", cudaGetErrorString(e));
    return launched("attention");
}

}  // namespace

// Up to three CTAs an SM, which run together; heads of 64 and more than 208 tokens leave room for two, and there up to two and a half.  Us
// in a chain of its own kind, this kernel and elsa_attention.cu's: 12 heads of 197 tokens, 1 image (156 CTAs) 2.6, 5.2, 2 images (312)
// 3.6, 5.2, 3 images (468) 5.7, 5.6, 4 images 6.4, 5.7, 8 images 9.6, 6.6; of 65 tokens, 6 images (360) 3.0, 3.9, 7 images (420) 3.6, 3.9; of
// 145 tokens, 3 images (360) 3.4, 4.8; 6 heads of 224 tokens, 4 images (336) 5.0, 5.1, 5 images (420) 5.3, 5.2.  In the encoder of
// DeiT-B an image's twelve take 36 of the 72 us they took (one image 499 -> 468 us, two images 593 -> 578).
bool attention_rows_suits(int images, int tokens, int heads, int head_dim, int sm_count)
{
    const int tk = (tokens + 15) / 16 * 16, smem = head_dim == 64 ? rows_smem<64>(tk) : rows_smem<32>(tk);
    const bool three = 3 * (smem + 1024 /* reserved for each CTA */) <= 228 * 1024;
    return 2LL * images * heads * ((tokens + kRows - 1) / kRows) <= (three ? 6LL : 5LL) * sm_count;
}

elsa_status launch_attention_rows(const uint16_t* qkv, int images, int tokens, int heads, int dim, elsa_dtype dtype, uint16_t* out,
                                  uint32_t* dev_status, cudaStream_t stream, const DeviceInfo& dev)
{
    RowsParams p;
    p.out = out;
    p.tokens = tokens; p.tk = (tokens + 15) / 16 * 16; p.dim = dim; p.heads = heads;
    p.row_tiles = (tokens + kRows - 1) / kRows;
    p.dev_status = dev_status;
    const int d = dim / heads;
    elsa_status st;
    if ((st = make_map_qkv(&p.map_q, qkv, images, tokens, dim, d, kRows, "q")) != ELSA_OK) return st;
    if ((st = make_map_qkv(&p.map_kv, qkv, images, tokens, dim, d, (uint32_t)p.tk, "k, v")) != ELSA_OK) return st;
    const bool bf = dtype == ELSA_BF16;
    if (d == 64) return bf ? launch<true, 64>(p, images, stream, dev) : launch<false, 64>(p, images, stream, dev);
    return bf ? launch<true, 32>(p, images, stream, dev) : launch<false, 32>(p, images, stream, dev);
}

}  // namespace elsa

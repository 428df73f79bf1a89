// Helper kernels of the masked linear's backward pass (ELSA, Alg. 2: the gradient is taken with respect to the
// sparse weights derived from the shared weight; for Y = X Wm^T + b that is dX = dY Wm, dW = mask .* dY^T X,
// db = column sums of dY).  The two contractions run on the dense tensor-core GEMM of the forward path, which
// wants both operands with the reduction index contiguous; these kernels bring the operands into that form:
//   transpose_packed  the packed weight as the transposed masked weight [in][out], for dX
//   mask_apply     zeroes the pruned positions of a dense [out][in] gradient in place, from the index stream
//   wgrad_finish   adds the ranges' sums of dW, rounds and masks; and the parts of db where dW's launch made them
//   colsum_partial column sums of dY over chunks of 512 rows where it did not (db alone, or more tiles than SM pairs);
//                  colsum_finish adds the chunks and rounds once
#include "elsa_pack_device.cuh"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace elsa {
namespace {

constexpr int kTile = 64;

template <bool kBf16>
__device__ __forceinline__ float to_float(uint16_t u)
{
    if constexpr (kBf16) return __uint_as_float((uint32_t)u << 16);
    else return __half2float(__ushort_as_half(u));
}

template <bool kBf16>
__device__ __forceinline__ uint16_t from_float(float f)
{
    if constexpr (kBf16) return __bfloat16_as_ushort(__float2bfloat16_rn(f));
    else return __half_as_ushort(__float2half_rn(f));
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void stmatrix_x4_transposed(uint32_t addr, const uint32_t (&r)[4])
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};"
                 :: "r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}

// dst [in][out] = the masked weight [out][in], transposed: one block per 64 x 64 tile (out % 8 == 0).  The tile is expanded
// from the packed form, 16 bytes of a row at a time, into shared memory, transposed there in 8 x 8 blocks (ldmatrix,
// stmatrix.trans; rows of 144 bytes keep both free of bank conflicts) and written with 16-byte stores.  A launch is a few
// MB and bound by latency (6 to 7 us between events), which is why the expansion, 6 to 10 us as a launch before this one,
// is part of it; NC: the level N, 0 for the others.
template <int M, int NC>
__global__ void __launch_bounds__(256)
transpose_packed_kernel(const uint16_t* __restrict__ vals, const uint32_t* __restrict__ idx, uint16_t* __restrict__ dst, int out, int in,
                        int N, int words_per_row)
{
    constexpr int kPitch = kTile + 8;   // values per shared-memory row
    __shared__ __align__(16) uint16_t tile_in[kTile][kPitch];
    __shared__ __align__(16) uint16_t tile_out[kTile][kPitch];
    pdl_wait_for_predecessors();
    pdl_release_successors();
    const int r0 = blockIdx.x * kTile, c0 = blockIdx.y * kTile;   // row tiles on x: their count has no 65535 limit
    const int t = threadIdx.x;
    // expand: 64 rows x 8 units of 8 positions (rows past out and columns past in as zeros)
    const size_t values_per_row = (size_t)(in / M) * (size_t)N;
    if constexpr (M == 16 || NC == M) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int slot = t + 256 * i, r = slot >> 3, v = slot & 7;
            uint4 u = make_uint4(0u, 0u, 0u, 0u);
            if (r0 + r < out && c0 + 8 * v < in) {
                const size_t row = (size_t)(r0 + r);
                if constexpr (NC == M) u = __ldg(reinterpret_cast<const uint4*>(vals + row * (size_t)in + c0 + 8 * v));
                else u = expand_unit16(vals + row * values_per_row, idx + row * (size_t)words_per_row, N, (c0 >> 3) + v);
            }
            *reinterpret_cast<uint4*>(&tile_in[r][8 * v]) = u;
        }
    } else {
        PackedUnit unit[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int slot = t + 256 * i, r = slot >> 3, v = slot & 7;
            if (r0 + r < out && c0 + 8 * v < in) {
                const size_t row = (size_t)(r0 + r);
                unit[i] = load_packed_unit<M, NC>(vals + row * values_per_row, idx + row * (size_t)words_per_row, N, (c0 >> 3) + v);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int slot = t + 256 * i, r = slot >> 3, v = slot & 7;
            uint4 u = make_uint4(0u, 0u, 0u, 0u);
            if (r0 + r < out && c0 + 8 * v < in) u = expand_packed_unit<M, NC>(unit[i], N);
            *reinterpret_cast<uint4*>(&tile_in[r][8 * v]) = u;
        }
    }
    __syncthreads();
    {
        // warp w transposes the eight 8 x 8 blocks of source rows 8w .. 8w + 7
        const int w = t >> 5, lane = t & 31;
        const uint32_t in_base = (uint32_t)__cvta_generic_to_shared(&tile_in[0][0]);
        const uint32_t out_base = (uint32_t)__cvta_generic_to_shared(&tile_out[0][0]);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int j = 4 * half + (lane >> 3);               // column block this lane addresses
            uint32_t r[4];
            ldmatrix_x4(in_base + (uint32_t)(((8 * w + (lane & 7)) * kPitch + 8 * j) * 2), r);
            stmatrix_x4_transposed(out_base + (uint32_t)(((8 * j + (lane & 7)) * kPitch + 8 * w) * 2), r);
        }
    }
    __syncthreads();
    // store: 64 dst rows (weight columns) x 8 vectors of 8 weight rows
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int slot = t + 256 * i;
        const int c = slot >> 3, v = slot & 7;
        if (c0 + c < in && r0 + 8 * v < out)
            *reinterpret_cast<uint4*>(dst + (size_t)(c0 + c) * (size_t)out + r0 + 8 * v) = *reinterpret_cast<const uint4*>(&tile_out[c][8 * v]);
    }
}

// partial[chunk][c] = sum of src[r][c] over the chunk's rows (kColsumRows per chunk).  A block covers 256 columns:
// 32 threads across (eight columns each, one 16-byte load per row) by 8 threads down; every thread adds its rows
// in ascending order, the eight row lanes are added in a fixed order, so the result does not depend on timing.
constexpr int kColsumRows = 512;

template <bool kBf16>
__global__ void __launch_bounds__(256)
colsum_partial_kernel(const uint16_t* __restrict__ src, int R, int C, float* __restrict__ partial)
{
    __shared__ float acc[8][256 + 8];
    pdl_wait_for_predecessors();
    pdl_release_successors();
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int c = blockIdx.y * 256 + 8 * tx;
    const int r_begin = blockIdx.x * kColsumRows;
    const int r_end = min(R, r_begin + kColsumRows);
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (c < C) {
        for (int r = r_begin + ty; r < r_end; r += 8) {
            const uint4 u = __ldg(reinterpret_cast<const uint4*>(src + (size_t)r * (size_t)C + c));
            const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                s[2 * q] += to_float<kBf16>((uint16_t)(w[q] & 0xffffu));
                s[2 * q + 1] += to_float<kBf16>((uint16_t)(w[q] >> 16));
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[ty][8 * tx + e] = s[e];
    __syncthreads();
    const int col = blockIdx.y * 256 + threadIdx.x;
    if (col < C) {
        float t = 0.f;
#pragma unroll
        for (int y = 0; y < 8; ++y) t += acc[y][threadIdx.x];
        partial[(size_t)blockIdx.x * (size_t)C + col] = t;
    }
}

// db[c] = round16(sum over parts of partial[part][c]), parts in ascending order.
template <bool kBf16>
__device__ __forceinline__ void sum_parts(const float* __restrict__ partial, int parts, int C, uint16_t* __restrict__ db, int block)
{
    const int c = block * 256 + (int)threadIdx.x;
    if (c >= C) return;
    float s = 0.f;
#pragma unroll 8
    for (int i = 0; i < parts; ++i) s += partial[(size_t)i * (size_t)C + c];
    db[c] = from_float<kBf16>(s);
}

template <bool kBf16>
__global__ void __launch_bounds__(256) colsum_finish_kernel(const float* __restrict__ partial, int parts, int C, uint16_t* __restrict__ db)
{
    pdl_wait_for_predecessors();
    pdl_release_successors();
    sum_parts<kBf16>(partial, parts, C, db, (int)blockIdx.x);
}

// One thread per group of M: keeps the N positions the index stream names, zeroes the rest.
template <int M>
__global__ void __launch_bounds__(256)
mask_apply_kernel(uint16_t* __restrict__ dW, const uint32_t* __restrict__ idx, int out, int in, int N, int words_per_row)
{
    constexpr int B = (M == 4) ? 2 : (M == 8) ? 3 : 4;
    pdl_wait_for_predecessors();
    pdl_release_successors();
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int groups_per_row = in / M;
    if (gid >= (long long)out * groups_per_row) return;
    const int o = (int)(gid / groups_per_row), g = (int)(gid % groups_per_row);
    const uint32_t* row = idx + (size_t)o * (size_t)words_per_row;
    uint32_t keep = 0;
    for (int t = 0; t < N; ++t) {
        const int bit = (g * N + t) * B;
        const int w = bit >> 5, sh = bit & 31;
        uint32_t f = row[w] >> sh;
        if (sh + B > 32) f |= row[w + 1] << (32 - sh);
        keep |= 1u << (f & (M - 1));
    }
    uint32_t* p = reinterpret_cast<uint32_t*>(dW + (size_t)o * (size_t)in + (size_t)g * M);
#pragma unroll
    for (int q = 0; q < M / 2; ++q) {
        const uint32_t m = ((keep >> (2 * q)) & 1u ? 0x0000ffffu : 0u) | ((keep >> (2 * q + 1)) & 1u ? 0xffff0000u : 0u);
        if (m != 0xffffffffu) p[q] &= m;
    }
}

// One thread per group of M weights: adds the ranges' fp32 sums in ascending order, rounds once, zeroes what the
// index stream does not keep (everything is kept when idx is NULL).  The first db_blocks blocks add the parts of db.
template <int M, bool kBf16>
__global__ void __launch_bounds__(256)
wgrad_finish_kernel(const float* __restrict__ partial, int splits, const uint32_t* __restrict__ idx, int out, int in, int N,
                    int words_per_row, uint16_t* __restrict__ dW, const float* __restrict__ db_sums, int db_parts,
                    uint16_t* __restrict__ db, int db_blocks)
{
    constexpr int B = (M == 4) ? 2 : (M == 8) ? 3 : 4;
    pdl_wait_for_predecessors();
    pdl_release_successors();
    if ((int)blockIdx.x < db_blocks) {
        sum_parts<kBf16>(db_sums, db_parts, out, db, (int)blockIdx.x);
        return;
    }
    const long long gid = (long long)((int)blockIdx.x - db_blocks) * 256 + threadIdx.x;
    const int groups_per_row = in / M;
    if (gid >= (long long)out * groups_per_row) return;
    const int o = (int)(gid / groups_per_row), g = (int)(gid % groups_per_row);
    uint32_t keep = 0xffffffffu;
    if (idx != nullptr) {
        keep = 0;
        const uint32_t* row = idx + (size_t)o * (size_t)words_per_row;
        for (int t = 0; t < N; ++t) {
            const int bit = (g * N + t) * B;
            const int w = bit >> 5, sh = bit & 31;
            uint32_t f = row[w] >> sh;
            if (sh + B > 32) f |= row[w + 1] << (32 - sh);
            keep |= 1u << (f & (M - 1));
        }
    }
    const size_t at = (size_t)o * (size_t)in + (size_t)g * M;
    const size_t plane = (size_t)out * (size_t)in;
    float acc[M];
#pragma unroll
    for (int q = 0; q < M / 4; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(partial + at + 4 * q);
        acc[4 * q] = v.x; acc[4 * q + 1] = v.y; acc[4 * q + 2] = v.z; acc[4 * q + 3] = v.w;
    }
    for (int s = 1; s < splits; ++s) {
#pragma unroll
        for (int q = 0; q < M / 4; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(partial + (size_t)s * plane + at + 4 * q);
            acc[4 * q] += v.x; acc[4 * q + 1] += v.y; acc[4 * q + 2] += v.z; acc[4 * q + 3] += v.w;
        }
    }
    uint32_t* dst = reinterpret_cast<uint32_t*>(dW + at);
#pragma unroll
    for (int q = 0; q < M / 2; ++q) {
        const uint32_t lo = (keep >> (2 * q)) & 1u ? from_float<kBf16>(acc[2 * q]) : 0u;
        const uint32_t hi = (keep >> (2 * q + 1)) & 1u ? from_float<kBf16>(acc[2 * q + 1]) : 0u;
        dst[q] = lo | (hi << 16);
    }
}

}  // namespace

elsa_status launch_transpose_packed(const uint16_t* vals, const uint32_t* idx, uint16_t* dst, int out, int in, int N, int M, cudaStream_t stream)
{
    const dim3 grid((unsigned)((out + kTile - 1) / kTile), (unsigned)((in + kTile - 1) / kTile));
    const int wpr = (int)index_words_per_row(in, N, M);
    auto* kernel = N == M   ? transpose_packed_kernel<16, 16>
                   : M == 16 ? transpose_packed_kernel<16, 0>
                   : M == 8  ? (N == 1   ? transpose_packed_kernel<8, 1>
                                : N == 2 ? transpose_packed_kernel<8, 2>
                                : N == 4 ? transpose_packed_kernel<8, 4>
                                         : transpose_packed_kernel<8, 0>)
                             : (N == 1 ? transpose_packed_kernel<4, 1> : N == 2 ? transpose_packed_kernel<4, 2> : transpose_packed_kernel<4, 0>);
    ProfileScope scope(ELSA_KERNEL_BACKWARD_FORMAT, stream);
    launch_pdl(kernel, grid, dim3(256), 0, stream, 1, vals, idx, dst, out, in, N, wpr);
    return launched("transpose_packed");
}

// db [C] = column sums of src [R][C]; partial: ceil(R / 512) * C floats of scratch.
elsa_status launch_colsum(const uint16_t* src, int R, int C, float* partial, uint16_t* db, elsa_dtype dtype, cudaStream_t stream)
{
    const int chunks = (R + kColsumRows - 1) / kColsumRows;
    {
        const dim3 grid((unsigned)chunks, (unsigned)((C + 255) / 256));
        ProfileScope scope(ELSA_KERNEL_BACKWARD_FORMAT, stream);
        if (dtype == ELSA_BF16) launch_pdl(colsum_partial_kernel<true>, grid, dim3(256), 0, stream, 1, src, R, C, partial);
        else launch_pdl(colsum_partial_kernel<false>, grid, dim3(256), 0, stream, 1, src, R, C, partial);
        elsa_status st = launched("colsum_partial");
        if (st != ELSA_OK) return st;
    }
    return launch_colsum_finish(partial, chunks, C, db, dtype, stream);
}

elsa_status launch_colsum_finish(const float* partial, int parts, int C, uint16_t* db, elsa_dtype dtype, cudaStream_t stream)
{
    const unsigned grid = (unsigned)((C + 255) / 256);
    ProfileScope scope(ELSA_KERNEL_BACKWARD_FORMAT, stream);
    if (dtype == ELSA_BF16) launch_pdl(colsum_finish_kernel<true>, dim3(grid), dim3(256), 0, stream, 1, partial, parts, C, db);
    else launch_pdl(colsum_finish_kernel<false>, dim3(grid), dim3(256), 0, stream, 1, partial, parts, C, db);
    return launched("colsum_finish");
}

elsa_status launch_wgrad_finish(const float* partial, int splits, const uint32_t* idx, int out, int in, int N, int M,
                                elsa_dtype dtype, uint16_t* dW, const float* db_sums, int db_parts, uint16_t* db, cudaStream_t stream)
{
    const long long groups = (long long)out * (in / M);
    const int db_blocks = db_parts > 0 ? (out + 255) / 256 : 0;
    const unsigned grid = (unsigned)((groups + 255) / 256 + db_blocks);
    const int wpr = (int)index_words_per_row(in, N, M);
    const uint32_t* ix = N == M ? nullptr : idx;
    const bool bf = dtype == ELSA_BF16;
    ProfileScope scope(ELSA_KERNEL_BACKWARD_FORMAT, stream);
#define ELSA_FINISH(MM)                                                                                                     \
    do {                                                                                                                  \
        if (bf) launch_pdl(wgrad_finish_kernel<MM, true>, dim3(grid), dim3(256), 0, stream, 1, partial, splits, ix, out, in, N, wpr, dW, db_sums, db_parts, db, db_blocks); \
        else launch_pdl(wgrad_finish_kernel<MM, false>, dim3(grid), dim3(256), 0, stream, 1, partial, splits, ix, out, in, N, wpr, dW, db_sums, db_parts, db, db_blocks);   \
    } while (0)
    if (M == 4) ELSA_FINISH(4);
    else if (M == 8) ELSA_FINISH(8);
    else ELSA_FINISH(16);
#undef ELSA_FINISH
    return launched("wgrad_finish");
}

elsa_status launch_mask_apply(uint16_t* dW, const uint32_t* idx, int out, int in, int N, int M, cudaStream_t stream)
{
    if (N == M) return ELSA_OK;
    const long long groups = (long long)out * (in / M);
    const unsigned grid = (unsigned)((groups + 255) / 256);
    const int wpr = (int)index_words_per_row(in, N, M);
    ProfileScope scope(ELSA_KERNEL_BACKWARD_FORMAT, stream);
    if (M == 4) launch_pdl(mask_apply_kernel<4>, dim3(grid), dim3(256), 0, stream, 1, dW, idx, out, in, N, wpr);
    else if (M == 8) launch_pdl(mask_apply_kernel<8>, dim3(grid), dim3(256), 0, stream, 1, dW, idx, out, in, N, wpr);
    else launch_pdl(mask_apply_kernel<16>, dim3(grid), dim3(256), 0, stream, 1, dW, idx, out, in, N, wpr);
    return launched("mask_apply");
}

}  // namespace elsa

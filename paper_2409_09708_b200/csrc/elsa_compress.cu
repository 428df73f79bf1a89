// N:M projection of weights and their compressed form (the inverse is in elsa_weight_images.cu).
//
// Sec. 3.1 / Eq. 1 of the ELSA paper with magnitude saliency (keep the N largest |w| of each group of M consecutive
// weights), written in the compressed form of Sec. 1 / Sec. 2 (kept values + one log2(M)-bit index each).  One kernel for
// one weight, a table of weights, or several levels of one weight: a block works on one (weight, level), whose N and M
// are compile-time constants for the levels in use.  A warp takes four segments of 32 units (a unit: 8 weights, or one
// group of 16), all loads requested first (one segment where that leaves SMs idle); a segment owns whole index words, which its lanes assemble with shuffles.
//
// A launch over a few MB is bound by latency, so every block runs at once and goes through memory once; a table of
// many weights is bound by integer issue and by HBM.  Against a persistent form that looked a table up per unit and
// assembled words with shared-memory atomics (us):
// the weights of DeiT-B's 48 linears (85M values) 91 -> 60, of Swin-B's 96 117 -> 68, of one DeiT-B block 16.2 -> 7.4; one
// 3072 x 768 weight to 1, 2, 4 and 8 of 8 16.4 -> 7.2.

#include "elsa_pack_device.cuh"

namespace elsa {
namespace {

constexpr int kThreads = kWarpsPerBlock * 32;

struct CompressItem {
    const uint16_t* W;
    uint16_t* vals;
    uint32_t* idx;
    int first_block;
    int N, M;
    // The weight as `rows` rows of `units` units.  Where a row's index bits fill whole words the rows follow one another
    // without padding and the weight is one long row.
    int rows, units, segs, words;     // segments and index words per row
    int out, in;
};

template <int kMax>
struct CompressTable {
    CompressItem item[kMax];
    int n;
};

// The kept values of a unit, two per word, and their index fields, first value lowest.
template <int M, int N, int kWords>
__device__ __forceinline__ void pick_unit(const uint32_t (&a)[kWords], uint32_t (&v)[4], uint32_t& fields)
{
    constexpr int B = M == 4 ? 2 : M == 8 ? 3 : 4, kGroups = M == 4 ? 2 : 1, kGroupWords = M / 2;
    v[0] = v[1] = v[2] = v[3] = 0u;
    fields = 0;
#pragma unroll
    for (int g = 0; g < kGroups; ++g) {
        uint32_t w[kGroupWords];
#pragma unroll
        for (int q = 0; q < kGroupWords; ++q) w[q] = a[g * kGroupWords + q];
        uint32_t keep;
        if constexpr (M == 16) {
            keep = keep_mask16<N>(w);
        } else {
            uint32_t h[M];
#pragma unroll
            for (int i = 0; i < M; ++i) h[i] = (w[i >> 1] >> (16 * (i & 1))) & 0xFFFFu;
            keep = keep_mask_sorted<M>(h, N);
        }
#pragma unroll
        for (int t = 0; t < N; ++t) {
            const uint32_t pos = t == N - 1 ? 31u - (uint32_t)__clz((int)keep) : (uint32_t)__ffs((int)keep) - 1u;
            keep &= keep - 1u;
            const int slot = g * N + t;
            v[slot >> 1] |= half_of(w, pos) << (16 * (slot & 1));
            fields |= pos << (slot * B);
        }
    }
}

// A segment's index words from its 32 lanes' kBits-bit fields: lane k of the first kBits returns word k.
template <int kBits>
__device__ __forceinline__ uint32_t assemble_words(uint32_t f, int lane)
{
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    if constexpr (kBits == 32) {
        return f;
    } else if constexpr (32 % kBits == 0) {            // 4, 8, 16: lanes merge into whole words
#pragma unroll
        for (int b = kBits, d = 1; b < 32; b *= 2, d *= 2) f |= __shfl_down_sync(kAll, f, d) << b;
        return __shfl_sync(kAll, f, (lane * (32 / kBits)) & 31);
    } else if constexpr (24 % kBits == 0) {            // 3, 6, 12: lanes merge into 24 bits, a word spans two of those
        constexpr int kLanes = 24 / kBits;
#pragma unroll
        for (int b = kBits, d = 1; b < 24; b *= 2, d *= 2) f |= __shfl_down_sync(kAll, f, d) << b;
        const int g = (32 * lane) / 24, off = (32 * lane) % 24;
        const uint32_t lo = __shfl_sync(kAll, f, (g * kLanes) & 31) & 0xFFFFFFu, hi = __shfl_sync(kAll, f, ((g + 1) * kLanes) & 31);
        return (lo >> off) | (hi << (24 - off));
    } else {
        uint32_t w = 0;
        const int first = (32 * lane) / kBits;
#pragma unroll
        for (int j = 0; j < (32 + kBits - 1) / kBits + 1; ++j) {
            const int l = first + j, sh = l * kBits - 32 * lane;
            const uint32_t x = __shfl_sync(kAll, f, l & 31);
            if (l < 32 && sh < 32) w |= sh >= 0 ? x << sh : x >> -sh;
        }
        return w;
    }
}

template <int M, int N, int kSegsPerWarp>
__device__ __forceinline__ void compress_block(const CompressItem& it, int block)
{
    constexpr int kSegsPerBlock = kWarpsPerBlock * kSegsPerWarp;
    constexpr int B = M == 4 ? 2 : M == 8 ? 3 : 4;
    constexpr int kUnit = M == 16 ? 16 : 8, kWords = kUnit / 2, kCount = kUnit / M * N, kBits = kCount * B;
    const int lane = threadIdx.x & 31;
    const int seg0 = block * kSegsPerBlock + (int)(threadIdx.x >> 5) * kSegsPerWarp;
    const int segs = it.segs, units = it.units, total = it.rows * segs;
    uint4 raw[kSegsPerWarp][kWords / 4];
    int row[kSegsPerWarp], seg[kSegsPerWarp];
#pragma unroll
    for (int i = 0; i < kSegsPerWarp; ++i) {
        row[i] = it.rows == 1 ? 0 : (seg0 + i) / segs;
        seg[i] = seg0 + i - row[i] * segs;
        if (seg0 + i < total && seg[i] * 32 + lane < units) {
            const uint4* src = reinterpret_cast<const uint4*>(it.W) + ((size_t)row[i] * units + (size_t)(seg[i] * 32 + lane)) * (kWords / 4);
#pragma unroll
            for (int q = 0; q < kWords / 4; ++q) raw[i][q] = __ldg(src + q);
        }
    }
#pragma unroll
    for (int i = 0; i < kSegsPerWarp; ++i) {
        if (seg0 + i >= total) return;
        const bool valid = seg[i] * 32 + lane < units;
        uint32_t v[4], fields = 0;
        if (valid) {
            uint32_t a[kWords];
#pragma unroll
            for (int q = 0; q < kWords / 4; ++q) { a[4 * q] = raw[i][q].x; a[4 * q + 1] = raw[i][q].y; a[4 * q + 2] = raw[i][q].z; a[4 * q + 3] = raw[i][q].w; }
            pick_unit<M, N>(a, v, fields);
            uint16_t* dst = it.vals + ((size_t)row[i] * units + (size_t)(seg[i] * 32 + lane)) * kCount;
            if constexpr (kCount == 8) *reinterpret_cast<uint4*>(dst) = make_uint4(v[0], v[1], v[2], v[3]);
            else if constexpr (kCount == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(v[0], v[1]);
            else if constexpr (kCount % 2 == 0) {
#pragma unroll
                for (int q = 0; q < kCount / 2; ++q) reinterpret_cast<uint32_t*>(dst)[q] = v[q];
            } else {
#pragma unroll
                for (int t = 0; t < kCount; ++t) dst[t] = (uint16_t)(v[t >> 1] >> (16 * (t & 1)));
            }
        }
        const uint32_t word = assemble_words<kBits>(fields, lane);
        const int at = seg[i] * kBits + lane;
        if (lane < kBits && at < it.words) it.idx[(size_t)row[i] * it.words + at] = word;
    }
}

// The dense level stores the weight as it is.
template <int kSegsPerWarp>
__device__ __forceinline__ void copy_block(const CompressItem& it, int block)
{
    constexpr int kSegsPerBlock = kWarpsPerBlock * kSegsPerWarp;
    const long long units = (long long)it.out * it.in / 8;
    const long long base = (long long)block * (kSegsPerBlock * 32) + threadIdx.x;
    uint4 v[kSegsPerWarp];
#pragma unroll
    for (int i = 0; i < kSegsPerWarp; ++i)
        if (base + i * kThreads < units) v[i] = __ldg(reinterpret_cast<const uint4*>(it.W) + base + i * kThreads);
#pragma unroll
    for (int i = 0; i < kSegsPerWarp; ++i)
        if (base + i * kThreads < units) reinterpret_cast<uint4*>(it.vals)[base + i * kThreads] = v[i];
}

// Any other level; kept out of line so that its registers do not count against the levels in use.
template <int M, int kSegsPerWarp>
__device__ __noinline__ void compress_block_any(const uint16_t* W, uint16_t* vals, uint32_t* idx, int out, int in, int N, int words_per_row,
                                                int block, uint32_t (*words)[kMaxIndexWordsPerSegment])
{
    constexpr int kSegsPerBlock = kWarpsPerBlock * kSegsPerWarp;
    const int segs_per_row = (in / M + 31) / 32;
    for (int i = 0; i < kSegsPerWarp; ++i) {
        const long long seg = (long long)block * kSegsPerBlock + (int)(threadIdx.x >> 5) * kSegsPerWarp + i;
        if (seg < (long long)out * segs_per_row) compress_segment<M>(W, in, N, vals, idx, segs_per_row, words_per_row, seg, words,
                                [N](const uint16_t (&w)[M]) { return keep_mask<M>(group_ranks<M>(w), N); });
    }
}

template <int kMax, int kSegs>
__global__ void __launch_bounds__(kThreads, 4) nm_compress_kernel(const __grid_constant__ CompressTable<kMax> t)
{
    __shared__ uint32_t words[kWarpsPerBlock][kMaxIndexWordsPerSegment];
    pdl_wait_for_predecessors();
    pdl_release_successors();
    int cur = 0;
    if constexpr (kMax > 1) {
        int hi = t.n - 1;
        while (cur < hi) {
            const int mid = (cur + hi + 1) >> 1;
            if (t.item[mid].first_block <= (int)blockIdx.x) cur = mid; else hi = mid - 1;
        }
    }
    const CompressItem& it = t.item[cur];
    const int block = (int)blockIdx.x - it.first_block;
    if (it.N == it.M) { copy_block<kSegs>(it, block); return; }
    switch (it.M * 32 + it.N) {
    case 4 * 32 + 1: compress_block<4, 1, kSegs>(it, block); break;
    case 4 * 32 + 2: compress_block<4, 2, kSegs>(it, block); break;
    case 4 * 32 + 3: compress_block<4, 3, kSegs>(it, block); break;
    case 8 * 32 + 1: compress_block<8, 1, kSegs>(it, block); break;
    case 8 * 32 + 2: compress_block<8, 2, kSegs>(it, block); break;
    case 8 * 32 + 3: compress_block<8, 3, kSegs>(it, block); break;
    case 8 * 32 + 4: compress_block<8, 4, kSegs>(it, block); break;
    case 16 * 32 + 1: compress_block<16, 1, kSegs>(it, block); break;
    case 16 * 32 + 2: compress_block<16, 2, kSegs>(it, block); break;
    case 16 * 32 + 4: compress_block<16, 4, kSegs>(it, block); break;
    case 16 * 32 + 8: compress_block<16, 8, kSegs>(it, block); break;
    default:
        if (it.M == 8) compress_block_any<8, kSegs>(it.W, it.vals, it.idx, it.out, it.in, it.N, it.words, block, words);
        else compress_block_any<16, kSegs>(it.W, it.vals, it.idx, it.out, it.in, it.N, it.words, block, words);
    }
}

// One weight at a level that the kernel above takes by its general form: kernels of their own, since the levels in use lose 5 % to
// more code beside them (4096 x 1024 to 1, 2, 3 and 4 of 8 14.9 -> 15.6 us).  4096 x 1024 at 5:8 15.2 -> 6.4 us, 3072 x 768 at
// 3:16 18.1 -> 9.3.
template <int N, int kSegs>
__global__ void __launch_bounds__(kThreads, 4) nm_compress_dense8_kernel(const __grid_constant__ CompressTable<1> t)
{
    pdl_wait_for_predecessors();
    pdl_release_successors();
    compress_block<8, N, kSegs>(t.item[0], (int)blockIdx.x);
}

__global__ void __launch_bounds__(kThreads, 4) nm_compress_any16_kernel(const __grid_constant__ CompressTable<1> t)
{
    __shared__ uint32_t words[kWarpsPerBlock][kMaxIndexWordsPerSegment];
    pdl_wait_for_predecessors();
    pdl_release_successors();
    const CompressItem& it = t.item[0];
    const int segs_per_row = (it.in / 16 + 31) / 32, N = it.N;
    const long long seg = (long long)blockIdx.x * kWarpsPerBlock + (int)(threadIdx.x >> 5);
    if (seg < (long long)it.out * segs_per_row)
        compress_segment<16>(it.W, it.in, N, it.vals, it.idx, segs_per_row, it.words, seg, words, [N](const uint16_t (&w)[16]) {
            uint32_t a[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) a[q] = (uint32_t)w[2 * q] | ((uint32_t)w[2 * q + 1] << 16);
            return keep_mask16_any(a, N);
        });
}

// Whether compress_block has the level.
bool fast_level(int N, int M) { return M == 4 || (M == 8 && N <= 4) || (M == 16 && (N == 1 || N == 2 || N == 4 || N == 8)); }

// Whether a launch of n weights is one for the kernels of single weights.
bool dense8(const CompressJob& j, int n) { return n == 1 && j.M == 8 && j.N >= 5 && j.N <= 7; }
bool any16(const CompressJob& j, int n) { return n == 1 && j.M == 16 && j.N < 16 && !fast_level(j.N, j.M); }

template <int kMax>
elsa_status launch_table(const CompressJob* jobs, int n, cudaStream_t stream)
{
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    CompressTable<kMax> t;      // on the stack: several threads may launch at once
    long long segs[kMax], total = 0;
    for (int i = 0; i < n; ++i) {
        const CompressJob& j = jobs[i];
        CompressItem& it = t.item[i];
        it.W = j.W; it.vals = j.vals; it.idx = j.idx; it.N = j.N; it.M = j.M; it.out = j.out; it.in = j.in;
        it.rows = j.out;
        it.words = (int)index_words_per_row(j.in, j.N, j.M);
        it.units = j.in / (j.M == 16 ? 16 : 8);
        const long long row_bits = (long long)(j.in / j.M) * j.N * index_bits(j.M);
        if (j.N == j.M || fast_level(j.N, j.M) || dense8(j, n)) {
            if (row_bits % 32 == 0 && (long long)j.out * it.units < (1ll << 30) && (long long)j.out * it.words < (1ll << 30)) {
                it.units *= j.out;
                it.words *= j.out;
                it.rows = 1;
            }
            it.segs = (it.units + 31) / 32;
        } else {
            it.segs = (j.in / j.M + 31) / 32;
        }
        segs[i] = j.N == j.M ? ((long long)j.out * j.in / 8 + 31) / 32 : (long long)it.rows * it.segs;
        total += segs[i];
    }
    // Four segments a warp keep four loads of a lane in flight; below two blocks an SM one segment a warp is quicker
    // (384 x 384: 18 blocks or 72; one weight at 2:8 2.3 against 1.6 us).
    const int per_warp = any16(jobs[0], n) || total < (long long)dev.sm_count * 2 * kWarpsPerBlock * 4 ? 1 : 4;
    int blocks = 0;
    for (int i = 0; i < n; ++i) {
        t.item[i].first_block = blocks;
        blocks += (int)((segs[i] + kWarpsPerBlock * per_warp - 1) / (kWarpsPerBlock * per_warp));
    }
    t.n = n;
    ProfileScope scope(ELSA_KERNEL_COMPRESS, stream);
    auto kernel = per_warp == 1 ? nm_compress_kernel<kMax, 1> : nm_compress_kernel<kMax, 4>;
    if constexpr (kMax == 1) {
        const int N = jobs[0].N;
        if (any16(jobs[0], n)) kernel = nm_compress_any16_kernel;
        else if (dense8(jobs[0], n))
            kernel = N == 5   ? (per_warp == 1 ? nm_compress_dense8_kernel<5, 1> : nm_compress_dense8_kernel<5, 4>)
                     : N == 6 ? (per_warp == 1 ? nm_compress_dense8_kernel<6, 1> : nm_compress_dense8_kernel<6, 4>)
                              : (per_warp == 1 ? nm_compress_dense8_kernel<7, 1> : nm_compress_dense8_kernel<7, 4>);
    }
    cudaError_t e = launch_pdl(kernel, dim3((unsigned)blocks), dim3(kThreads),
                               0, stream, 1, t);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(ELSA_ERR_CUDA, "launch of nm_compress failed: %s", cudaGetErrorString(e));
    }
    return launched("nm_compress");
}

}  // namespace

elsa_status launch_compress_jobs(const CompressJob* jobs, int n, cudaStream_t stream)
{
    constexpr int kMost = 256;       // items per launch (kernel parameters are limited to 32 KB)
    for (int at = 0; at < n; at += kMost) {
        const int count = n - at < kMost ? n - at : kMost;
        const elsa_status st = count == 1   ? launch_table<1>(jobs + at, count, stream)
                               : count <= 8 ? launch_table<8>(jobs + at, count, stream)
                                            : launch_table<kMost>(jobs + at, count, stream);
        if (st != ELSA_OK) return st;
    }
    return ELSA_OK;
}

elsa_status launch_compress(const uint16_t* W, int out, int in, int N, int M, uint16_t* vals, uint32_t* idx, cudaStream_t stream)
{
    const CompressJob j = {W, vals, idx, out, in, N, M};
    return launch_compress_jobs(&j, 1, stream);
}

}  // namespace elsa

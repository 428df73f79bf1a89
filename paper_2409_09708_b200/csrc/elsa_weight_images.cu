// Weight images: what the tensor-core kernels read in place of the packed weight (Sec. 2, Fig. 2 of the ELSA paper: the
// indices give each kept value's position).  Four kinds, from the packed form or from a dense shared weight projected
// onto its level on the way (Sec. 3.1):
//   IMAGE_UNPACK, IMAGE_MASK        the dense masked weight [out][in]
//   IMAGE_SP24, IMAGE_MASK_SP24     N <= 2: two values per aligned chunk of 4 and the metadata of the 2:4 sparse MMA
// One kernel for any number of weights: a block of 256 threads works on one weight, at a level known at compile time
// for the common ones, and every thread has the loads of all its units in flight before it expands the first.  The
// images are a few MB, so what bounds a launch is latency, and what bounds a large table is the traffic through L2.
// Against one thread per 8 or 16 positions with a loop over the kept values: image and GEMM of 3152 x 768 -> 3072 at 2:4
// 20.6 -> 17.1 us back to back (the 2-of-4 image about 6 -> 2.5), of 197 x 768 -> 2304 on the dense image 8.2 -> 7.5; the
// four images of a DeiT-B block in one launch 22 -> 12.6 us between events.  A thread has four dense units, or one where
// those would be fewer than two blocks for an SM: 256 x 256 2.1 -> 1.5 us, 768 x 768 2.3 -> 1.7, 512 x 2048 at 8:16
// 4.6 -> 3.1; from there up both take the same.

#include <vector>

#include "elsa_sp24_device.cuh"

namespace elsa {
namespace {

constexpr int kImageThreads = 256;
constexpr int kMostUnits = 4;             // dense images: units of 8 positions per thread, or one (see launch_images)
constexpr long long kUnitsMost = 1ll << 31;   // of one image in a launch: a block's first unit and its last fit 32 bits

struct ImageItem {
    const uint16_t* src;
    const uint32_t* idx;
    uint16_t* dst;
    uint16_t* meta;
    int first_block;
    int out, in, N, M, words_per_row, kind, layout;
    int rounds;                           // a block works on this many runs of its threads' units, one after the other
    uint32_t magic;                       // floor(2^32 / d) of the division that finds a thread's row, see split_by
    int k_blocks, steps;                  // 2-of-4 forms: metadata blocks along K, K steps of 32 per block (2 or 4)
};

template <int kMax>
struct ImageTable {
    ImageItem item[kMax];
    int n;
};

// n / d and n % d for any 32-bit n: the product's high half is one short at most.
__device__ __forceinline__ uint32_t split_by(uint32_t n, uint32_t d, uint32_t magic, uint32_t& rest)
{
    uint32_t q = __umulhi(n, magic);
    rest = n - q * d;
    if (rest >= d) { ++q; rest -= d; }
    return q;
}

// ---------------------------------------------------------------- dense images

// load(unit, row, unit of the row)
template <typename Raw, int kUnits, typename Load, typename Finish>
__device__ __forceinline__ void dense_image_block(const ImageItem& it, int block, Load load, Finish finish)
{
    const uint32_t units_per_row = (uint32_t)it.in >> 3, units = (uint32_t)it.out * units_per_row;
#pragma unroll 1
    for (int round = 0; round < it.rounds; ++round) {
        const uint32_t base = (uint32_t)(block * it.rounds + round) * (kImageThreads * kUnits) + threadIdx.x;
        Raw raw[kUnits];
        int half[kUnits];
#pragma unroll
        for (int i = 0; i < kUnits; ++i) {
            // a unit past the end reads the last one: no branch stands between the loads
            const uint32_t unit = min(base + (uint32_t)(i * kImageThreads), units - 1u);
            uint32_t u;
            const uint32_t row = split_by(unit, units_per_row, it.magic, u);
            half[i] = (int)(u & 1u);
            raw[i] = load((size_t)unit, row, (int)u);
        }
#pragma unroll
        for (int i = 0; i < kUnits; ++i) {
            const uint32_t unit = base + (uint32_t)(i * kImageThreads);
            if (unit >= units) break;
            reinterpret_cast<uint4*>(it.dst)[unit] = finish(raw[i], half[i]);
        }
    }
}

template <int M, int NC, int kUnits>
__device__ __forceinline__ void unpack_block(const ImageItem& it, int block)
{
    const int N = it.N, wpr = it.words_per_row, count = (8 / M) * (NC ? NC : N);
    dense_image_block<PackedUnit, kUnits>(
        it, block, [&](size_t unit, uint32_t row, int u) { return load_packed_values<M, NC>(it.src + unit * count, it.idx + (size_t)row * wpr, N, u); },
        [&](const PackedUnit& p, int) { return expand_packed_unit<M, NC>(p, N); });
}

// The same for groups of 16, one a thread: load(group, row, group of the row), finish(raw) -> Group16.  (By halves of a group every
// thread read and ranked the whole of it: image and GEMM of 3152 x 1024 -> 4096 at 4:16 from the shared weight 53 us, 24.7 like this.
// From the packed form the halves stay quicker where the launch leaves SMs idle: 2048 x 512 at 8:16 and below about 1 us.)
template <typename Raw, int kGroups, typename Load, typename Finish>
__device__ __forceinline__ void group16_image_block(const ImageItem& it, int block, Load load, Finish finish)
{
    const uint32_t groups_per_row = (uint32_t)it.in >> 4, groups = (uint32_t)it.out * groups_per_row;
#pragma unroll 1
    for (int round = 0; round < it.rounds; ++round) {
        const uint32_t base = (uint32_t)(block * it.rounds + round) * (kImageThreads * kGroups) + threadIdx.x;
        Raw raw[kGroups];
#pragma unroll
        for (int i = 0; i < kGroups; ++i) {
            const uint32_t group = min(base + (uint32_t)(i * kImageThreads), groups - 1u);
            uint32_t g;
            const uint32_t row = split_by(group, groups_per_row, it.magic, g);
            raw[i] = load((size_t)group, row, (int)g);
        }
#pragma unroll
        for (int i = 0; i < kGroups; ++i) {
            const uint32_t group = base + (uint32_t)(i * kImageThreads);
            if (group >= groups) break;
            const Group16 d = finish(raw[i]);
            reinterpret_cast<uint4*>(it.dst)[2 * (size_t)group] = d.a;
            reinterpret_cast<uint4*>(it.dst)[2 * (size_t)group + 1] = d.b;
        }
    }
}

// ---------------------------------------------------------------- 2-of-4 images

// A thread has 16 positions of image rows m and m + 8 of a block of 16 rows: the two share a metadata word.  Eight lanes
// cover the eight row pairs, four groups of lanes four consecutive 16-position segments.
// Image row o holds feature o_src: in the permuted forms (Sp24Layout) row r of a block of 32 holds feature
// 8 * (r % 4) + r / 4.  Rows are padded to 128 for the metadata (zero), to 32 for the values.
template <int M, int N, bool kMask>
__device__ __forceinline__ void sp24_block(const ImageItem& it, int block)
{
    const int out = it.out, in = it.in, steps = it.steps, k_blocks = it.k_blocks;
    const int segs = k_blocks * steps * 2;                         // per row, padding included
    const int seg_groups = segs >> 2;
#pragma unroll 1
    for (int round = 0; round < it.rounds; ++round) {
        const int slot = (block * it.rounds + round) * (kImageThreads / 32) + (int)(threadIdx.x >> 5);      // (16 rows, 4 segments) of this warp
        uint32_t group;
        const int rows16 = (int)split_by((uint32_t)slot, (uint32_t)seg_groups, it.magic, group);
        if (rows16 >= (out + 127) / 128 * 8) return;
        const int lane = threadIdx.x & 31;
        const int seg = (int)group * 4 + (lane >> 3);
        const int o0 = rows16 * 16 + (lane & 7);
        const int k0 = seg * 16;
        int src_row[2];
        Segment s[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int o = o0 + 8 * i, r = o & 31;
            src_row[i] = it.layout != SP24_ROWS ? (o & ~31) | (8 * (r & 3) + (r >> 2)) : o;
            if (src_row[i] < out && k0 < in) {
                if constexpr (kMask) {
                    const uint4* g = reinterpret_cast<const uint4*>(it.src + (size_t)src_row[i] * in + k0);
                    s[i] = pick_segment<M, N>(__ldg(g), __ldg(g + 1));
                } else {
                    s[i] = load_segment<M, N>(it.src + (size_t)src_row[i] * (in / M * N), it.idx + (size_t)src_row[i] * it.words_per_row, seg);
                }
            }
        }
        uint32_t word = 0;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            uint32_t nib = 0x4444u;                                    // four empty chunks
            if (src_row[i] < out && k0 < in) v = sp24_words<M, N>(s[i], nib);
            word |= nib << (16 * i);
            if (k0 < in && src_row[i] < ((out + 31) & ~31)) {
                const int o = o0 + 8 * i;
                size_t at = (size_t)o * (size_t)in + (size_t)k0;       // byte offset of (row o, k0) in the row-major forms
                if (it.layout == SP24_TILED)
                    at = (size_t)(o >> 5) * 32 * (size_t)in + (size_t)(k0 >> 8) * 8192 + (size_t)((((k0 & 255) >> 4) * 32 + (o & 31)) * 16);
                *reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(it.dst) + at) = v;
            }
        }
        // metadata: block (128 features, k block) -> tensor-memory lane -> 4 words, one per K step of 32; a block of 64 k
        // leaves the last two zero
        const int kb = seg / (2 * steps), step = (seg >> 1) % steps, k1 = seg & 1;
        const int tm_lane = (lane & 7) + 8 * k1 + 16 * (rows16 & 7);
        uint32_t* meta = reinterpret_cast<uint32_t*>(it.meta) + (((size_t)(rows16 >> 3) * k_blocks + kb) * 128 + tm_lane) * 4 + step;
        meta[0] = word;
        if (steps == 2) meta[2] = 0u;
    }
}

// Whether a dense image's unit is a whole group of 16, one a thread, instead of 8 positions.
bool in_groups16(const ImageJob& j, int units_per_thread) { return j.M == 16 && (j.kind == IMAGE_MASK || (j.kind == IMAGE_UNPACK && j.N != 16 && units_per_thread > 1)); }

// Blocks of a weight.
int image_blocks(const ImageJob& j, int units_per_thread, int rounds)
{
    if (j.kind == IMAGE_UNPACK || j.kind == IMAGE_MASK) {
        const bool groups16 = in_groups16(j, units_per_thread);
        const long long units = (long long)j.out * (groups16 ? j.in / 16 : j.in / 8);
        const long long per_block = (long long)kImageThreads * (groups16 ? 1 : units_per_thread) * rounds;
        return (int)((units + per_block - 1) / per_block);
    }
    const long long segs = (long long)((j.in + j.block_k - 1) / j.block_k) * (j.block_k / 32) * 2;
    const long long warps = (long long)((j.out + 127) / 128 * 8) * (segs / 4);
    const long long per_block = (long long)(kImageThreads / 32) * rounds;
    return (int)((warps + per_block - 1) / per_block);
}

template <int kMax, int kUnits>
__global__ void __launch_bounds__(kImageThreads, 4) weight_image_kernel(const __grid_constant__ ImageTable<kMax> t)
{
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
    const ImageItem& it = t.item[cur];
    const int block = (int)blockIdx.x - it.first_block;
    const int N = it.N, M = it.M;
    if (it.kind == IMAGE_SP24) {
        if (M == 4) { if (N == 2) sp24_block<4, 2, false>(it, block); else sp24_block<4, 1, false>(it, block); }
        else if (M == 8) { if (N == 2) sp24_block<8, 2, false>(it, block); else sp24_block<8, 1, false>(it, block); }
        else { if (N == 2) sp24_block<16, 2, false>(it, block); else sp24_block<16, 1, false>(it, block); }
    } else if (it.kind == IMAGE_MASK_SP24) {
        if (M == 4) { if (N == 2) sp24_block<4, 2, true>(it, block); else sp24_block<4, 1, true>(it, block); }
        else if (M == 8) { if (N == 2) sp24_block<8, 2, true>(it, block); else sp24_block<8, 1, true>(it, block); }
        else { if (N == 2) sp24_block<16, 2, true>(it, block); else sp24_block<16, 1, true>(it, block); }
    } else if (it.kind == IMAGE_UNPACK) {
        if (N == M) {
            dense_image_block<uint4, kUnits>(it, block, [&](size_t unit, uint32_t, int) { return __ldg(reinterpret_cast<const uint4*>(it.src) + unit); },
                                             [](const uint4& v, int) { return v; });
        } else if (M == 8) {
            if (N == 1) unpack_block<8, 1, kUnits>(it, block);
            else if (N == 2) unpack_block<8, 2, kUnits>(it, block);
            else if (N == 3) unpack_block<8, 3, kUnits>(it, block);
            else if (N == 4) unpack_block<8, 4, kUnits>(it, block);
            else unpack_block<8, 0, kUnits>(it, block);
        } else if (M == 4) {
            if (N == 1) unpack_block<4, 1, kUnits>(it, block);
            else if (N == 2) unpack_block<4, 2, kUnits>(it, block);
            else unpack_block<4, 3, kUnits>(it, block);
        } else {
            const int vpr = it.in / 16 * N, wpr = it.words_per_row;
            if constexpr (kUnits == 1)      // a small launch: threads before instructions
                dense_image_block<uint2, 1>(
                    it, block, [](size_t, uint32_t row, int u) { return make_uint2(row, (uint32_t)u); },
                    [&](const uint2& at, int) { return expand_unit16(it.src + (size_t)at.x * vpr, it.idx + (size_t)at.x * wpr, N, (int)at.y); });
            else group16_image_block<PackedGroup16, 1>(
                it, block, [&](size_t, uint32_t row, int g) { return load_packed_group16(it.src + (size_t)row * vpr, it.idx + (size_t)row * wpr, N, g); },
                [&](const PackedGroup16& p) { return expand_packed_group16(p, N); });
        }
    } else {
        if (M == 16) {
            group16_image_block<Group16, 1>(
                it, block,
                [&](size_t group, uint32_t, int) {
                    const uint4* g = reinterpret_cast<const uint4*>(it.src) + 2 * group;
                    return Group16{__ldg(g), __ldg(g + 1)};
                },
                [&](const Group16& g) { return mask_group16(g, N); });
        } else {
            dense_image_block<uint4, kUnits>(it, block, [&](size_t unit, uint32_t, int) { return __ldg(reinterpret_cast<const uint4*>(it.src) + unit); },
                                             [&](const uint4& v, int) { return M == 8 ? mask_unit<8>(v, v, 0, N) : mask_unit<4>(v, v, 0, N); });
        }
    }
}

template <int kMax, int kUnits>
elsa_status launch_table(const ImageJob* jobs, int n, int rounds, cudaStream_t stream)
{
    ImageTable<kMax> t;      // on the stack: several threads may launch at once
    int blocks = 0;
    for (int i = 0; i < n; ++i) {
        const ImageJob& j = jobs[i];
        ImageItem& it = t.item[i];
        it.src = j.src; it.idx = j.idx; it.dst = j.dst; it.meta = (uint16_t*)j.meta;
        it.first_block = blocks;
        it.out = j.out; it.in = j.in; it.N = j.N; it.M = j.M; it.kind = j.kind; it.layout = j.layout;
        it.words_per_row = (int)index_words_per_row(j.in, j.N, j.M);
        it.k_blocks = (j.in + j.block_k - 1) / j.block_k;
        it.steps = j.block_k / 32;
        const bool dense = j.kind == IMAGE_UNPACK || j.kind == IMAGE_MASK;
        const uint32_t d = dense ? (uint32_t)j.in / (in_groups16(j, kUnits) ? 16 : 8) : (uint32_t)(it.k_blocks * it.steps * 2) >> 2;
        it.magic = d == 1 ? 0xFFFFFFFFu : (uint32_t)((1ull << 32) / d);
        it.rounds = rounds;
        blocks += image_blocks(j, kUnits, rounds);
    }
    t.n = n;
    const int k = n > 1 || jobs[0].kind == IMAGE_MASK ? ELSA_KERNEL_WEIGHT_IMAGES : jobs[0].kind == IMAGE_UNPACK ? ELSA_KERNEL_UNPACK : ELSA_KERNEL_NM_TO_SP24;
    ProfileScope scope(k, stream);
    cudaError_t e = launch_pdl(weight_image_kernel<kMax, kUnits>, dim3((unsigned)blocks), dim3(kImageThreads), 0, stream, 1, t);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(ELSA_ERR_CUDA, "launch of the weight images failed: %s", cudaGetErrorString(e));
    }
    return launched("weight images");
}

}  // namespace

elsa_status launch_images(const ImageJob* jobs, int n, cudaStream_t stream)
{
    // A dense image's units are counted in 32 bits: a weight of more goes in runs of rows, each with its part of the packed form.
    for (int i = 0; i < n; ++i) {
        const ImageJob& j = jobs[i];
        const long long rows = kUnitsMost / (j.in / 8);
        if ((j.kind != IMAGE_UNPACK && j.kind != IMAGE_MASK) || j.out <= rows) continue;
        const bool packed = j.kind == IMAGE_UNPACK;
        const size_t src_row = packed ? values_per_row(j.in, j.N, j.M) : (size_t)j.in, idx_row = index_words_per_row(j.in, j.N, j.M);
        std::vector<ImageJob> cut(jobs, jobs + i);
        for (long long r = 0; r < j.out; r += rows) {
            ImageJob part = j;
            part.src = j.src + (size_t)r * src_row;
            part.idx = j.idx != nullptr ? j.idx + (size_t)r * idx_row : nullptr;
            part.dst = j.dst + (size_t)r * (size_t)j.in;
            part.out = (int)(j.out - r < rows ? j.out - r : rows);
            cut.push_back(part);
        }
        cut.insert(cut.end(), jobs + i + 1, jobs + n);
        return launch_images(cut.data(), (int)cut.size(), stream);
    }
    DeviceInfo dev;
    const elsa_status dev_st = device_info(&dev);
    if (dev_st != ELSA_OK) return dev_st;
    constexpr int kMost = 256;       // items per launch (kernel parameters are limited to 32 KB)
    for (int at = 0; at < n; at += kMost) {
        const int count = n - at < kMost ? n - at : kMost;
        int blocks = 0;
        for (int i = 0; i < count; ++i) {      // groups of 16 count as what their positions are elsewhere
            const int b = image_blocks(jobs[at + i], kMostUnits, 1);
            blocks += in_groups16(jobs[at + i], kMostUnits) ? (b + 1) / 2 : b;
        }
        const bool spread = blocks < 2 * dev.sm_count;
        // A block costs a few thousand cycles before its first load, so where there are many waves of them they take three
        // runs each: 48 DeiT-B weights at 2:8 to dense images 51 -> 46 us, to 2-of-4 ones 60 -> 55; one block's four
        // weights 4.4 to 4.9 with two runs, 5.0 with four.
        const int rounds = blocks >= 32 * dev.sm_count ? 3 : 1;
        const elsa_status st =
            count == 1   ? (spread ? launch_table<1, 1>(jobs + at, count, 1, stream) : launch_table<1, kMostUnits>(jobs + at, count, rounds, stream))
            : count <= 8 ? (spread ? launch_table<8, 1>(jobs + at, count, 1, stream) : launch_table<8, kMostUnits>(jobs + at, count, rounds, stream))
                         : launch_table<kMost, kMostUnits>(jobs + at, count, rounds, stream);
        if (st != ELSA_OK) return st;
    }
    return ELSA_OK;
}

elsa_status launch_unpack(const uint16_t* vals, const uint32_t* idx, int out, int in, int N, int M, uint16_t* Wm, cudaStream_t stream)
{
    ImageJob j;
    j.kind = IMAGE_UNPACK; j.src = vals; j.idx = idx; j.dst = Wm; j.out = out; j.in = in; j.N = N; j.M = M;
    return launch_images(&j, 1, stream);
}

elsa_status launch_nm_to_sp24(const uint16_t* vals, const uint32_t* idx, int out, int in, int N, int M, int block_k, int layout,
                              uint16_t* a_img, uint8_t* meta, cudaStream_t stream)
{
    ImageJob j;
    j.kind = IMAGE_SP24; j.src = vals; j.idx = idx; j.dst = a_img; j.meta = meta; j.out = out; j.in = in; j.N = N; j.M = M;
    j.layout = layout; j.block_k = block_k;
    return launch_images(&j, 1, stream);
}

}  // namespace elsa

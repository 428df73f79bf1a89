// Device code shared by the kernels that read or write the packed weight: the choice of the kept positions of a group
// (Sec. 3.1 / Eq. 1 of the ELSA paper), the general form of packing (the levels in use have their own in elsa_compress.cu),
// and the expansion of eight consecutive positions from the packed form (Sec. 1 / Sec. 2) or from a dense weight.
#pragma once

#include "elsa_internal.h"

namespace elsa {
namespace {

constexpr int kWarpsPerBlock = 8;
constexpr int kMaxIndexWordsPerSegment = 64;  // 32 groups x N*b bits, N*b <= 60 for N < M <= 16

template <int M>
__device__ __forceinline__ void load_group(const uint16_t* p, uint16_t (&w)[M])
{
    if constexpr (M == 4) {
        uint2 v = *reinterpret_cast<const uint2*>(p);
        w[0] = v.x & 0xFFFF; w[1] = v.x >> 16; w[2] = v.y & 0xFFFF; w[3] = v.y >> 16;
    } else {
#pragma unroll
        for (int q = 0; q < M / 8; ++q) {
            uint4 v = reinterpret_cast<const uint4*>(p)[q];
            w[8 * q + 0] = v.x & 0xFFFF; w[8 * q + 1] = v.x >> 16;
            w[8 * q + 2] = v.y & 0xFFFF; w[8 * q + 3] = v.y >> 16;
            w[8 * q + 4] = v.z & 0xFFFF; w[8 * q + 5] = v.z >> 16;
            w[8 * q + 6] = v.w & 0xFFFF; w[8 * q + 7] = v.w >> 16;
        }
    }
}

// Ranks of the M magnitudes of one group, 4 bits each: rank_i = #{j : |w_j| > |w_i|} + #{j < i : |w_j| == |w_i|}
// (larger magnitude first, lower position first among equals).  Magnitudes are compared as the 15 low
// bits of the pattern.  The level N keeps exactly the elements with rank < N, for every N at once.
template <int M>
__device__ __forceinline__ unsigned long long group_ranks(const uint16_t (&w)[M])
{
    unsigned long long ranks = 0;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        const uint32_t ki = w[i] & 0x7FFFu;
        int rank = 0;
#pragma unroll
        for (int j = 0; j < M; ++j) {
            const uint32_t kj = w[j] & 0x7FFFu;
            rank += (kj > ki) || (j < i && kj == ki);
        }
        ranks |= (unsigned long long)rank << (4 * i);
    }
    return ranks;
}

template <int M>
__device__ __forceinline__ uint32_t keep_mask(unsigned long long ranks, int N)
{
    uint32_t keep = 0;
#pragma unroll
    for (int i = 0; i < M; ++i) keep |= (uint32_t)((int)((ranks >> (4 * i)) & 15ull) < N) << i;
    return keep;
}

// One warp compresses 32 consecutive groups of one row, one group per lane, at any level N < M: the form for the levels
// that have none of their own (elsa_compress.cu); keep_of: the mask of a group.  The 32 groups own exactly N*b whole index words of the row's
// bitstream, so the warp assembles its words in shared memory and writes them with one coalesced store.
template <int M, typename Keep>
__device__ __forceinline__ void compress_segment(const uint16_t* __restrict__ W, int in, int N, uint16_t* __restrict__ vals,
                                                 uint32_t* __restrict__ idx, int segs_per_row, int words_per_row, long long seg_id,
                                                 uint32_t (*words)[kMaxIndexWordsPerSegment], Keep keep_of)
{
    constexpr int B = (M == 4) ? 2 : (M == 8) ? 3 : 4;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;

    const int o = (int)(seg_id / segs_per_row);
    const int seg = (int)(seg_id % segs_per_row);
    const int groups_per_row = in / M;
    const int g = seg * 32 + lane;
    const int seg_words = N * B;  // index words this segment owns

    for (int k = lane; k < seg_words; k += 32) words[warp][k] = 0;
    __syncwarp();
    if (g < groups_per_row) {
        uint16_t w[M];
        load_group<M>(W + (size_t)o * in + (size_t)g * M, w);
        const uint32_t keep = keep_of(w);
        uint16_t* v = vals + (size_t)o * ((size_t)groups_per_row * N) + (size_t)g * N;
        unsigned long long fields = 0;
        int t = 0;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            if ((keep >> i) & 1u) {
                v[t] = w[i];
                fields |= (unsigned long long)i << (t * B);
                ++t;
            }
        }
        const int bit0 = lane * seg_words;  // bit offset of this group's fields in the segment
        const int w0 = bit0 >> 5, sh = bit0 & 31;
        // up to 60 bits shifted by up to 31: three words at most
        const uint32_t lo = (uint32_t)(fields << sh);
        const uint32_t mid = (uint32_t)(fields >> (32 - sh));
        const uint32_t hi = sh ? (uint32_t)(fields >> (64 - sh)) : 0u;
        // a zero part may lie past the segment's last word and is skipped
        if (lo) atomicOr(&words[warp][w0], lo);
        if (mid) atomicOr(&words[warp][w0 + 1], mid);
        if (hi) atomicOr(&words[warp][w0 + 2], hi);
    }
    __syncwarp();
    const int first = seg * seg_words;
    uint32_t* row = idx + (size_t)o * words_per_row;
    for (int k = lane; k < seg_words && first + k < words_per_row; k += 32) row[first + k] = words[warp][k];
    __syncwarp();
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

__device__ __forceinline__ void sort2_desc(uint32_t& a, uint32_t& b)
{
    const uint32_t hi = max(a, b), lo = min(a, b);
    a = hi; b = lo;
}

// Keep mask of one group: bit i set iff position i is among the N kept.  h[] are the 16-bit patterns.
template <int M>
__device__ __forceinline__ uint32_t keep_mask_sorted(const uint32_t (&h)[M], int N)
{
    constexpr int S = (M == 4) ? 2 : 3;
    uint32_t k[M], s[M];
#pragma unroll
    for (int i = 0; i < M; ++i) { k[i] = ((h[i] & 0x7FFFu) << S) | (uint32_t)(M - 1 - i); s[i] = k[i]; }
    if constexpr (M == 8) {
        // The levels of the ViT tables need less than a full sort.  Keys are unique and carry their position
        // in the low bits, so the one or two largest keys name the kept positions directly; for N = 4 two
        // sorted halves give the 4th largest without merging them.
        if (N <= 2) {
            sort2_desc(s[0], s[1]); sort2_desc(s[2], s[3]); sort2_desc(s[4], s[5]); sort2_desc(s[6], s[7]);
            // top two of each half from two sorted pairs, then of the whole group
            const uint32_t a0 = max(s[0], s[2]), a1 = max(min(s[0], s[2]), max(s[1], s[3]));
            const uint32_t b0 = max(s[4], s[6]), b1 = max(min(s[4], s[6]), max(s[5], s[7]));
            const uint32_t top = max(a0, b0), second = max(min(a0, b0), max(a1, b1));
            uint32_t keep = 1u << (7u - (top & 7u));
            if (N == 2) keep |= 1u << (7u - (second & 7u));
            return keep;
        }
        if (N == 4) {
            sort2_desc(s[0], s[1]); sort2_desc(s[2], s[3]); sort2_desc(s[4], s[5]); sort2_desc(s[6], s[7]);
            sort2_desc(s[0], s[2]); sort2_desc(s[1], s[3]); sort2_desc(s[4], s[6]); sort2_desc(s[5], s[7]);
            sort2_desc(s[1], s[2]); sort2_desc(s[5], s[6]);
            // i elements of one half and j of the other lie above min(a_i, b_j): with i + j = 2 it is at most the
            // 4th largest, and so are a_3 and b_3 (a half that supplies all four); the largest candidate is it
            const uint32_t thr4 = max(max(max(s[3], s[7]), min(s[0], s[6])), max(min(s[1], s[5]), min(s[2], s[4])));
            uint32_t keep4 = 0;
#pragma unroll
            for (int i = 0; i < M; ++i) keep4 |= (k[i] >= thr4 ? 1u : 0u) << i;
            return keep4;
        }
    }
    if constexpr (M == 4) {
        sort2_desc(s[0], s[1]); sort2_desc(s[2], s[3]);
        sort2_desc(s[0], s[2]); sort2_desc(s[1], s[3]);
        sort2_desc(s[1], s[2]);
    } else {
        sort2_desc(s[0], s[1]); sort2_desc(s[2], s[3]); sort2_desc(s[4], s[5]); sort2_desc(s[6], s[7]);
        sort2_desc(s[0], s[2]); sort2_desc(s[1], s[3]); sort2_desc(s[4], s[6]); sort2_desc(s[5], s[7]);
        sort2_desc(s[1], s[2]); sort2_desc(s[5], s[6]);
        sort2_desc(s[0], s[4]); sort2_desc(s[1], s[5]); sort2_desc(s[2], s[6]); sort2_desc(s[3], s[7]);
        sort2_desc(s[2], s[4]); sort2_desc(s[3], s[5]);
        sort2_desc(s[1], s[2]); sort2_desc(s[3], s[4]); sort2_desc(s[5], s[6]);
    }
    uint32_t thr = s[0];
#pragma unroll
    for (int t = 1; t < M; ++t) thr = (N > t) ? s[t] : thr;      // the N-th largest key
    uint32_t keep = 0;
#pragma unroll
    for (int i = 0; i < M; ++i) keep |= (k[i] >= thr ? 1u : 0u) << i;
    return keep;
}

// The 16 bits at position `pos` of consecutive positions packed two to a word.
template <int kWords>
__device__ __forceinline__ uint32_t half_of(const uint32_t (&a)[kWords], uint32_t pos)
{
    uint32_t w;
    if constexpr (kWords == 2) w = pos & 2u ? a[1] : a[0];
    else if constexpr (kWords == 4) w = pos & 4u ? (pos & 2u ? a[3] : a[2]) : (pos & 2u ? a[1] : a[0]);
    else {
        const uint32_t lo = pos & 4u ? (pos & 2u ? a[3] : a[2]) : (pos & 2u ? a[1] : a[0]);
        const uint32_t hi = pos & 4u ? (pos & 2u ? a[7] : a[6]) : (pos & 2u ? a[5] : a[4]);
        w = pos & 8u ? hi : lo;
    }
    return (pos & 1u ? w >> 16 : w) & 0xFFFFu;
}

// Keep mask of a group of 16 (words of two positions).  The even and the odd positions' magnitudes are sorted side
// by side, two to an instruction; the N-th largest of the two sorted lists A, B is the largest of the minima of A's i-th
// and B's (N - i)-th.  What exceeds it is kept, and of what equals it the lowest positions that are still needed.  (768 x
// 768 at 2:16 1.8 us against 5.8 by ranks; groups of 8 and 4 are 5 to 20 % quicker by keep_mask_sorted.)
__device__ __forceinline__ void sort_halves16(const uint32_t (&a)[8], uint32_t (&k)[8], uint32_t (&s)[8])
{
#pragma unroll
    for (int q = 0; q < 8; ++q) s[q] = k[q] = a[q] & 0x7FFF7FFFu;
    auto sort2 = [&](int x, int y) {
        const uint32_t hi = __vmaxu2(s[x], s[y]), lo = __vminu2(s[x], s[y]);
        s[x] = hi; s[y] = lo;
    };
    sort2(0, 1); sort2(2, 3); sort2(4, 5); sort2(6, 7);
    sort2(0, 2); sort2(1, 3); sort2(4, 6); sort2(5, 7);
    sort2(1, 2); sort2(5, 6);
    sort2(0, 4); sort2(1, 5); sort2(2, 6); sort2(3, 7);
    sort2(2, 4); sort2(3, 5);
    sort2(1, 2); sort2(3, 4); sort2(5, 6);
}

// The N-th largest magnitude of the two sorted lists.
template <int N>
__device__ __forceinline__ uint32_t threshold16(const uint32_t (&s)[8])
{
    static_assert(N >= 1 && N <= 15, "levels below the dense one");
    constexpr int kFirst = N > 8 ? N - 8 : 0, kLast = N < 8 ? N : 8;      // how many of the N may come from A
    uint32_t thr = 0;
#pragma unroll
    for (int i = kFirst; i <= kLast; ++i) {       // i of A and N - i of B lie at or above the candidate
        const uint32_t x = i > 0 ? s[i > 0 ? i - 1 : 0] & 0xFFFFu : 0xFFFFu, y = i < N ? s[i < N ? N - i - 1 : 0] >> 16 : 0xFFFFu;
        thr = max(thr, min(x, y));
    }
    return thr;
}

__device__ __forceinline__ uint32_t keep_above16(const uint32_t (&k)[8], uint32_t thr, int N)
{
    const uint32_t thr2 = thr | (thr << 16);
    uint32_t above = 0, least = 0;       // magnitudes > thr, >= thr (15-bit values: a borrow clears the half's top bit)
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const uint32_t g = ~((thr2 | 0x80008000u) - k[q]) & 0x80008000u, e = ((k[q] | 0x80008000u) - thr2) & 0x80008000u;
        above |= (((g >> 15) | (g >> 30)) & 3u) << (2 * q);
        least |= (((e >> 15) | (e >> 30)) & 3u) << (2 * q);
    }
    uint32_t equal = least & ~above;
    int need = N - __popc(above);
    if (__popc(equal) == need) return least;
    uint32_t keep = above;
    for (; need > 0; --need) {
        keep |= equal & (0u - equal);
        equal &= equal - 1u;
    }
    return keep;
}

template <int N>
__device__ __forceinline__ uint32_t keep_mask16(const uint32_t (&a)[8])
{
    uint32_t k[8], s[8];
    sort_halves16(a, k, s);
    return keep_above16(k, threshold16<N>(s), N);
}

// The same for a level known at run time.
__device__ __forceinline__ uint32_t keep_mask16_any(const uint32_t (&a)[8], int N)
{
    uint32_t k[8], s[8], thr;
    sort_halves16(a, k, s);
    switch (N) {
    case 1: thr = threshold16<1>(s); break;
    case 2: thr = threshold16<2>(s); break;
    case 3: thr = threshold16<3>(s); break;
    case 4: thr = threshold16<4>(s); break;
    case 5: thr = threshold16<5>(s); break;
    case 6: thr = threshold16<6>(s); break;
    case 7: thr = threshold16<7>(s); break;
    case 8: thr = threshold16<8>(s); break;
    case 9: thr = threshold16<9>(s); break;
    case 10: thr = threshold16<10>(s); break;
    case 11: thr = threshold16<11>(s); break;
    case 12: thr = threshold16<12>(s); break;
    case 13: thr = threshold16<13>(s); break;
    case 14: thr = threshold16<14>(s); break;
    default: thr = threshold16<15>(s); break;
    }
    return keep_above16(k, thr, N);
}

// ---- eight consecutive positions of a packed row as one 16-byte unit (groups of 4: two groups, groups of 8: one),
// in two halves so that a caller can have the loads of several units in flight before it expands the first.
struct PackedUnit {
    uint32_t v[4];      // the unit's kept values in order, two per word
    uint32_t fields;    // their index fields, first value lowest
};

// NC: the level's N as a compile-time constant (0 = take `N_runtime`).  N < M.  Reads go past L1, which is not known to be
// clean of older contents while a predecessor kernel still runs (see `early` in elsa_linear_small.cu).
template <int M, int NC>
__device__ __forceinline__ PackedUnit load_packed_values(const uint16_t* __restrict__ v, const uint32_t* __restrict__ idx_row,
                                                         int N_runtime, int unit)
{
    static_assert(M == 4 || M == 8, "groups of 16 hold two units: expand_unit16");
    constexpr int B = M == 4 ? 2 : 3;
    const int N = NC ? NC : N_runtime;
    const int count = (8 / M) * N;              // values of the unit
    PackedUnit p;
    p.v[0] = p.v[1] = p.v[2] = p.v[3] = 0u;
    if ((count & 3) == 0) {                     // 4 values at most (8 would be the dense level)
        const uint2 t = __ldcg(reinterpret_cast<const uint2*>(v));
        p.v[0] = t.x; p.v[1] = t.y;
    } else if ((count & 1) == 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (q < (count >> 1)) p.v[q] = __ldcg(reinterpret_cast<const uint32_t*>(v) + q);
    } else {
#pragma unroll
        for (int t = 0; t < 7; ++t)
            if (t < count) p.v[t >> 1] |= (uint32_t)__ldcg(v + t) << (16 * (t & 1));
    }
    const int bit0 = unit * count * B, w0 = bit0 >> 5, sh = bit0 & 31;
    const uint32_t lo = __ldcg(idx_row + w0);
    const uint32_t hi = (sh + count * B > 32) ? __ldcg(idx_row + w0 + 1) : 0u;
    p.fields = __funnelshift_r(lo, hi, sh);
    return p;
}

// The same from the start of the row's values.
template <int M, int NC>
__device__ __forceinline__ PackedUnit load_packed_unit(const uint16_t* __restrict__ vals_row, const uint32_t* __restrict__ idx_row,
                                                       int N_runtime, int unit)
{
    return load_packed_values<M, NC>(vals_row + (size_t)unit * (size_t)((8 / M) * (NC ? NC : N_runtime)), idx_row, N_runtime, unit);
}

// shl that gives 0 for shifts of 32 and more (negative ones included)
__device__ __forceinline__ uint32_t shl_or_zero(uint32_t v, uint32_t s)
{
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
    return r;
}

// Up to two values (the halves of w) at the positions of a group of 8 or 4: byte-permute selectors that start as "zero
// byte" (bytes of the permute's second operand) and get the value's two bytes at its position, 8 selector bits apiece.
template <bool kTwo>
__device__ __forceinline__ uint4 place_in_8(uint32_t w, uint32_t fields)
{
    const uint32_t a0 = (fields << 3) & 0x38u, a1 = fields & 0x38u;
    uint32_t lo = 0x44444444u ^ shl_or_zero(0x54u, a0), hi = 0x44444444u ^ shl_or_zero(0x54u, a0 - 32u);
    if constexpr (kTwo) {
        lo ^= shl_or_zero(0x76u, a1);
        hi ^= shl_or_zero(0x76u, a1 - 32u);
    }
    return make_uint4(prmt(w, 0u, lo), prmt(w, 0u, lo >> 16), prmt(w, 0u, hi), prmt(w, 0u, hi >> 16));
}

// kTwo: both halves of w; otherwise its low (kHigh: high) half alone.
template <bool kTwo, bool kHigh>
__device__ __forceinline__ uint2 place_in_4(uint32_t w, uint32_t fields)
{
    uint32_t sel = 0x44444444u ^ ((kHigh ? 0x76u : 0x54u) << ((fields << 3) & 0x18u));
    if constexpr (kTwo) sel ^= 0x76u << ((fields << 1) & 0x18u);
    return make_uint2(prmt(w, 0u, sel), prmt(w, 0u, sel >> 16));
}

// The unit's eight positions: values at theirs, +0.0 elsewhere.  The common levels place one or two values per permute;
// the others split the values into a plane of low bytes and one of high bytes, scatter those by byte permutes
// (selector nibble of a position = slot of its value; slot 7 is zero because fewer than eight values are kept) and
// re-interleave.
template <int M, int NC>
__device__ __forceinline__ uint4 expand_packed_unit(const PackedUnit& p, int N_runtime)
{
    if constexpr (M == 8 && NC == 1) return place_in_8<false>(p.v[0], p.fields);
    if constexpr (M == 8 && NC == 2) return place_in_8<true>(p.v[0], p.fields);
    if constexpr (M == 8 && NC == 4) {
        const uint4 a = place_in_8<true>(p.v[0], p.fields), b = place_in_8<true>(p.v[1], p.fields >> 6);
        return make_uint4(a.x | b.x, a.y | b.y, a.z | b.z, a.w | b.w);
    }
    if constexpr (M == 4 && NC == 1) {
        const uint2 a = place_in_4<false, false>(p.v[0], p.fields), b = place_in_4<false, true>(p.v[0], p.fields >> 2);
        return make_uint4(a.x, a.y, b.x, b.y);
    }
    if constexpr (M == 4 && NC == 2) {
        const uint2 a = place_in_4<true, false>(p.v[0], p.fields), b = place_in_4<true, false>(p.v[1], p.fields >> 4);
        return make_uint4(a.x, a.y, b.x, b.y);
    }
    constexpr int B = M == 4 ? 2 : 3;
    const int N = NC ? NC : N_runtime;
    uint32_t sel = 0x77777777u;
#pragma unroll
    for (int t = 0; t < 7; ++t)
        if (t < (8 / M) * N) {
            uint32_t pos = (p.fields >> (t * B)) & (uint32_t)(M - 1);
            if (M == 4 && t >= N) pos += 4u;
            sel ^= (uint32_t)(7 ^ t) << (4u * pos);      // positions are distinct: the nibble is still 7
        }
    const uint32_t l0 = prmt(p.v[0], p.v[1], 0x6420u), l1 = prmt(p.v[2], p.v[3], 0x6420u);
    const uint32_t h0 = prmt(p.v[0], p.v[1], 0x7531u), h1 = prmt(p.v[2], p.v[3], 0x7531u);
    const uint32_t pl03 = prmt(l0, l1, sel & 0xFFFFu), pl47 = prmt(l0, l1, sel >> 16);
    const uint32_t ph03 = prmt(h0, h1, sel & 0xFFFFu), ph47 = prmt(h0, h1, sel >> 16);
    return make_uint4(prmt(pl03, ph03, 0x5140u), prmt(pl03, ph03, 0x7362u), prmt(pl47, ph47, 0x5140u), prmt(pl47, ph47, 0x7362u));
}

// ---- a whole group of 16 of a packed row, N < 16, in the same two halves
struct PackedGroup16 {
    uint32_t w[8];                 // kept values in order, two per word
    unsigned long long fields;
};

__device__ __forceinline__ PackedGroup16 load_packed_group16(const uint16_t* __restrict__ vals_row, const uint32_t* __restrict__ idx_row, int N, int g)
{
    PackedGroup16 p;
    const int bit0 = g * N * 4, w0 = bit0 >> 5, sh = bit0 & 31;
    unsigned long long fields = __ldcg(idx_row + w0);
    if (sh + 4 * N > 32) fields |= (unsigned long long)__ldcg(idx_row + w0 + 1) << 32;
    fields >>= sh;
    if (sh + 4 * N > 64) fields |= (unsigned long long)__ldcg(idx_row + w0 + 2) << (64 - sh);
    p.fields = fields;
    const uint16_t* v = vals_row + (size_t)g * N;
    if ((N & 3) == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint2 t = 4 * q < N ? __ldcg(reinterpret_cast<const uint2*>(v) + q) : make_uint2(0u, 0u);
            p.w[2 * q] = t.x; p.w[2 * q + 1] = t.y;
        }
    } else if ((N & 1) == 0) {
#pragma unroll
        for (int q = 0; q < 8; ++q) p.w[q] = 2 * q < N ? __ldcg(reinterpret_cast<const uint32_t*>(v) + q) : 0u;
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            p.w[q] = 2 * q < N ? (uint32_t)__ldcg(v + 2 * q) : 0u;
            if (2 * q + 1 < N) p.w[q] |= (uint32_t)__ldcg(v + 2 * q + 1) << 16;
        }
    }
    return p;
}

struct Group16 { uint4 a, b; };    // sixteen positions

__device__ __forceinline__ Group16 expand_packed_group16(const PackedGroup16& p, int N)
{
    uint32_t d[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
    for (int t = 0; t < 15; ++t) {
        if (t >= N) break;
        const uint32_t pos = (uint32_t)(p.fields >> (4 * t)) & 15u, x = (p.w[t >> 1] >> (16 * (t & 1))) & 0xFFFFu, s = 16u * (pos & 3u);
        const uint32_t lo = shl_or_zero(x, s), hi = shl_or_zero(x, s - 32u);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if ((pos >> 2) == (uint32_t)q) { d[2 * q] |= lo; d[2 * q + 1] |= hi; }
    }
    return Group16{make_uint4(d[0], d[1], d[2], d[3]), make_uint4(d[4], d[5], d[6], d[7])};
}

// A dense group of 16 projected onto level N:16.
__device__ __forceinline__ Group16 mask_group16(const Group16& g, int N)
{
    uint32_t a[8] = {g.a.x, g.a.y, g.a.z, g.a.w, g.b.x, g.b.y, g.b.z, g.b.w};
    const uint32_t keep = keep_mask16_any(a, N);
#pragma unroll
    for (int q = 0; q < 8; ++q) a[q] &= ((keep >> (2 * q)) & 1u ? 0xFFFFu : 0u) | ((keep >> (2 * q + 1)) & 1u ? 0xFFFF0000u : 0u);
    return Group16{make_uint4(a[0], a[1], a[2], a[3]), make_uint4(a[4], a[5], a[6], a[7])};
}

// A unit of a packed row with groups of 16: half of group unit / 2.
__device__ __forceinline__ uint4 expand_unit16(const uint16_t* __restrict__ vals_row, const uint32_t* __restrict__ idx_row, int N, int unit)
{
    const int g = unit >> 1, bit0 = g * N * 4, w0 = bit0 >> 5, sh = bit0 & 31;
    unsigned long long fields = __ldcg(idx_row + w0);
    if (sh + 4 * N > 32) fields |= (unsigned long long)__ldcg(idx_row + w0 + 1) << 32;
    fields >>= sh;
    if (sh + 4 * N > 64) fields |= (unsigned long long)__ldcg(idx_row + w0 + 2) << (64 - sh);
    // every value is asked for before the first is placed (one at a time each waited for the one before)
    const uint16_t* v = vals_row + (size_t)g * N;
    uint32_t w[8];
    if ((N & 1) == 0) {
#pragma unroll
        for (int q = 0; q < 8; ++q) w[q] = 2 * q < N ? __ldcg(reinterpret_cast<const uint32_t*>(v) + q) : 0u;
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            w[q] = 2 * q < N ? (uint32_t)__ldcg(v + 2 * q) : 0u;
            if (2 * q + 1 < N) w[q] |= (uint32_t)__ldcg(v + 2 * q + 1) << 16;
        }
    }
    unsigned long long lo = 0, hi = 0;
#pragma unroll
    for (int t = 0; t < 16; ++t) {
        if (t >= N) break;
        const uint32_t pos = (uint32_t)(fields >> (4 * t)) & 15u;
        const unsigned long long x = (unsigned long long)((w[t >> 1] >> (16 * (t & 1))) & 0xFFFFu) << (16u * (pos & 3u));
        if ((int)(pos >> 3) == (unit & 1)) {
            if (pos & 4u) hi |= x; else lo |= x;
        }
    }
    return make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
}

// Out of line: the few-rows kernel's other levels lose 2 % to the sort in their code (125 x 768 -> 192 at 2:4 6.21 us, 6.08).
__device__ __noinline__ uint32_t keep_mask16_call(uint4 a, uint4 b, int N)
{
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    return keep_mask16_any(w, N);
}

// Eight consecutive positions of a DENSE row projected onto level N:M, from the 16 bytes of the unit (groups of 16:
// from the whole group w, w16, with `half` saying which eight are wanted).
template <int M>
__device__ __forceinline__ uint4 mask_unit(const uint4& w, const uint4& w16, int half, int N)
{
    uint32_t keep = 0, a[4] = {w.x, w.y, w.z, w.w};
    if constexpr (M == 16) {
        keep = keep_mask16_call(w, w16, N) >> (8 * half);
        if (half) { a[0] = w16.x; a[1] = w16.y; a[2] = w16.z; a[3] = w16.w; }
    } else {
#pragma unroll
        for (int gl = 0; gl < 8 / M; ++gl) {
            uint32_t h[M];
#pragma unroll
            for (int i = 0; i < M; ++i) h[i] = (a[(gl * M + i) >> 1] >> (16 * (i & 1))) & 0xFFFFu;
            keep |= keep_mask_sorted<M>(h, N) << (gl * M);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] &= ((keep >> (2 * q)) & 1u ? 0xFFFFu : 0u) | ((keep >> (2 * q + 1)) & 1u ? 0xFFFF0000u : 0u);
    return make_uint4(a[0], a[1], a[2], a[3]);
}

}  // namespace
}  // namespace elsa

// From kept values and index fields (N <= 2 per group) to what the 2:4 sparse MMA reads: two values per aligned chunk of 4 and
// the metadata nibble of their positions.  Shared by the kernel that builds weight images and the one that expands the packed
// weight on its way to tensor memory.
#pragma once

#include "elsa_pack_device.cuh"

namespace elsa {
namespace {

// The kept values (N <= 2 per group) of 16 consecutive positions of a row, in order, and their index fields.
struct Segment {
    uint32_t v[4];
    uint32_t fields;
};

template <int M, int N>
__device__ __forceinline__ Segment load_segment(const uint16_t* __restrict__ vals_row, const uint32_t* __restrict__ idx_row, int seg)
{
    constexpr int B = M == 4 ? 2 : M == 8 ? 3 : 4;
    constexpr int count = 16 / M * N;
    Segment s;
    s.v[0] = s.v[1] = s.v[2] = s.v[3] = 0u;
    const uint16_t* v = vals_row + (size_t)seg * count;
    if constexpr (count == 8) {
        const uint4 t = __ldg(reinterpret_cast<const uint4*>(v));
        s.v[0] = t.x; s.v[1] = t.y; s.v[2] = t.z; s.v[3] = t.w;
    } else if constexpr (count == 4) {
        const uint2 t = __ldg(reinterpret_cast<const uint2*>(v));
        s.v[0] = t.x; s.v[1] = t.y;
    } else if constexpr (count == 2) {
        s.v[0] = __ldg(reinterpret_cast<const uint32_t*>(v));
    } else {
        s.v[0] = __ldg(v);
    }
    const int bit0 = seg * count * B, w0 = bit0 >> 5, sh = bit0 & 31;
    const uint32_t lo = __ldg(idx_row + w0);
    const uint32_t hi = (sh + count * B > 32) ? __ldg(idx_row + w0 + 1) : 0u;
    s.fields = __funnelshift_r(lo, hi, sh);
    return s;
}

// The same from 16 dense positions (words a[8]), projected onto level N:M (the N of largest magnitude, lowest position
// first among equals).
template <int M, int N>
__device__ __forceinline__ Segment pick_segment(const uint4& x, const uint4& y)
{
    const uint32_t a[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    Segment s;
    s.v[0] = s.v[1] = s.v[2] = s.v[3] = 0u;
    s.fields = 0;
    if constexpr (M == 16) {
        const uint32_t keep = keep_mask16<N>(a);
        const uint32_t p0 = (uint32_t)__ffs((int)keep) - 1u, p1 = 31u - (uint32_t)__clz((int)keep);
        s.v[0] = half_of(a, p0);
        s.fields = p0;
        if constexpr (N == 2) {
            s.v[0] |= half_of(a, p1) << 16;
            s.fields |= p1 << 4;
        }
    } else if constexpr (M == 8) {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const uint32_t w[4] = {a[4 * g], a[4 * g + 1], a[4 * g + 2], a[4 * g + 3]};
            uint32_t h[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) h[i] = (w[i >> 1] >> (16 * (i & 1))) & 0xFFFFu;
            const uint32_t keep = keep_mask_sorted<8>(h, N);
            const uint32_t p0 = (uint32_t)__ffs((int)keep) - 1u, p1 = 31u - (uint32_t)__clz((int)keep);
            if constexpr (N == 1) {
                s.v[0] |= half_of(w, p0) << (16 * g);
                s.fields |= p0 << (3 * g);
            } else {
                s.v[g] = half_of(w, p0) | (half_of(w, p1) << 16);
                s.fields |= (p0 | (p1 << 3)) << (6 * g);
            }
        }
    } else {
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const uint32_t w[2] = {a[2 * g], a[2 * g + 1]};
            const uint32_t h[4] = {w[0] & 0xFFFFu, w[0] >> 16, w[1] & 0xFFFFu, w[1] >> 16};
            const uint32_t keep = keep_mask_sorted<4>(h, N);
            const uint32_t p0 = (uint32_t)__ffs((int)keep) - 1u, p1 = 31u - (uint32_t)__clz((int)keep);
            const uint32_t v0 = half_of(w, p0), v1 = half_of(w, p1);
            if constexpr (N == 1) {
                s.v[g >> 1] |= v0 << (16 * (g & 1));
                s.fields |= p0 << (2 * g);
            } else {
                s.v[g] = v0 | (v1 << 16);
                s.fields |= (p0 | (p1 << 2)) << (4 * g);
            }
        }
    }
    return s;
}

// Groups of 8: how the kept values (one or two in a word) make the two words of a group, as selectors of byte permutes against
// zero, and the two metadata nibbles.  Indexed by the group's fields, two values first, then at 64 one.
// (Compares and selects for every chunk: 3072 x 768 at 2:8 3.1 us, with the table 2.7.)
struct alignas(8) Sp24Entry { uint32_t select, nibbles; };
struct Sp24Table {
    Sp24Entry e[64 + 8];
};
constexpr Sp24Table make_sp24_table()
{
    Sp24Table t{};
    for (int i = 0; i < 72; ++i) {
        const int n = i < 64 ? 2 : 1, p[2] = {i & 7, (i >> 3) & 7};
        uint32_t select = 0, nibbles = 0;
        for (int c = 0; c < 2; ++c) {
            uint32_t sel = 0x4444u, nib = 4u;                              // an empty chunk: zeros, positions 0 and 1
            const bool first = p[0] >> 2 == c, second = n == 2 && p[1] >> 2 == c;
            if (first && second) {
                sel = 0x3210u;
                nib = (uint32_t)(p[0] & 3) | (uint32_t)(p[1] & 3) << 2;
            } else if (first || second) {
                const uint32_t value = first ? 0x10u : 0x32u, l = (uint32_t)(first ? p[0] : p[1]) & 3u;
                sel = l == 3u ? value << 8 | 0x44u : 0x4400u | value;      // position 3 comes second, behind a zero at 0
                nib = l == 3u ? 0xCu : l | 0xCu;
            }
            select |= sel << (16 * c);
            nibbles |= nib << (4 * c);
        }
        t.e[i].select = select;
        t.e[i].nibbles = nibbles;
    }
    return t;
}
__device__ const Sp24Table kSp24Table = make_sp24_table();

// The 2-of-4 form of a segment: per aligned chunk of 4 two values with ascending positions i0 < i1 and the metadata
// nibble i0 | i1 << 2.  A chunk with one kept value takes position 3 as the second (0 as the first where the value itself
// is at 3), one with none takes 0 and 1; the values borrowed there are zero.
template <int M, int N>
__device__ __forceinline__ uint4 sp24_words(const Segment& s, uint32_t& nibbles)
{
    uint32_t w[4], nib = 0;
    // one value (low half of v) at position l of chunk c, if `here`
    auto single = [&](bool here, uint32_t v, uint32_t l, int c) {
        w[c] = here ? (l == 3u ? v << 16 : v) : 0u;
        nib |= (here ? (l == 3u ? 0xCu : (l | 0xCu)) : 4u) << (4 * c);
    };
    if constexpr (M == 4 && N == 2) {
        w[0] = s.v[0]; w[1] = s.v[1]; w[2] = s.v[2]; w[3] = s.v[3];
        nib = s.fields & 0xFFFFu;
    } else if constexpr (M == 8) {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const uint32_t f = (s.fields >> (g * N * 3)) & (N == 2 ? 63u : 7u), v = N == 2 ? s.v[g] : s.v[0] >> (16 * g);
            const uint2 e = __ldg(reinterpret_cast<const uint2*>(&kSp24Table.e[(N == 2 ? 0u : 64u) + f]));
            w[2 * g] = prmt(v, 0u, e.x & 0xFFFFu);
            w[2 * g + 1] = prmt(v, 0u, e.x >> 16);
            nib |= e.y << (8 * g);
        }
    } else if constexpr (M == 4) {
#pragma unroll
        for (int c = 0; c < 4; ++c) single(true, (s.v[c >> 1] >> (16 * (c & 1))) & 0xFFFFu, (s.fields >> (2 * c)) & 3u, c);
    } else if constexpr (N == 1) {              // one group of 16
        const uint32_t p0 = s.fields & 15u;
#pragma unroll
        for (int c = 0; c < 4; ++c) single((p0 >> 2) == (uint32_t)c, s.v[0], p0 & 3u, c);
    } else {
        // Selectors of byte permutes as with groups of 8, made by arithmetic: four empty chunks, and what each value changes in
        // its chunk's selector and nibble.  Two values of one chunk take its halves in order, as 0x3210 says.
        // (Compares and selects for every chunk, on the weight-stationary kernel: 12608 x 512 -> 512 at 2:16 13.2 us, like this 9.7.)
        const uint32_t p0 = s.fields & 15u, p1 = (s.fields >> 4) & 15u, l0 = p0 & 3u, l1 = p1 & 3u, at0 = p0 & 12u, at1 = p1 & 12u;
        const bool same = at0 == at1;
        const uint64_t select = 0x4444444444444444ull ^ ((uint64_t)(l0 == 3u ? 0x5400u : 0x0054u) << (4u * at0)) ^
                                ((uint64_t)(l1 == 3u || same ? 0x7600u : 0x0076u) << (4u * at1));
        const uint32_t lo = (uint32_t)select, hi = (uint32_t)(select >> 32);
        w[0] = prmt(s.v[0], 0u, lo & 0xFFFFu);
        w[1] = prmt(s.v[0], 0u, lo >> 16);
        w[2] = prmt(s.v[0], 0u, hi & 0xFFFFu);
        w[3] = prmt(s.v[0], 0u, hi >> 16);
        const uint32_t n0 = same ? (l0 | l1 << 2) ^ 4u : l0 == 3u ? 8u : 8u | l0, n1 = same ? 0u : l1 == 3u ? 8u : 8u | l1;
        nib = 0x4444u ^ (n0 << at0) ^ (n1 << at1);
    }
    nibbles = nib;
    return make_uint4(w[0], w[1], w[2], w[3]);
}

}  // namespace
}  // namespace elsa

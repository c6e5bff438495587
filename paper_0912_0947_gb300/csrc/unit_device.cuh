// unit_device.cuh -- units of 16 pixels (16*CH consecutive bytes) shared by the
// paper layout's kernels and the k-bit stream's: where they start in a cover
// and a stego at any addresses, where their plane bytes sit, and the byte
// moves between a unit's words and its 16 plane bytes.
#pragma once

#include "internal.cuh"

namespace stego {

// Where the plane bytes of a unit sit, as byte_perm selectors and masks: a unit's
// bytes are held as words w[0 .. 4*CH), its 16 plane bytes gathered into (or
// pairs taken from) four words, byte t%4 of word t/4 for pixel t.  With one
// channel they are the words themselves; with three, four pixels' plane bytes
// are bytes ph, ph + 3, ph + 6 and ph + 9 of three words; with four, byte ph of
// each word.  Selectors made once per launch (or cover) cost one byte_perm in
// twelve words more than compile-time positions, and one kernel serves every
// plane and every alignment of it.
struct PlaneSel {
    uint32_t get0, get1;         // gather: words 0 and 1, then word 2
    uint32_t put0, put1, put2;   // scatter: three channels into words 0, 1, 2; four:
                                 // byte t of a word by put0 | t << put1
    uint32_t mask0, mask1, mask2; // the low two bits of the plane bytes
};

__host__ __device__ inline PlaneSel make_sel(uint32_t ch, uint32_t ph)
{
    PlaneSel s{};
    if (ch == 3) {
        s.get0 = ph == 0 ? 0x0630u : ph == 1 ? 0x0741u : 0x0052u;
        s.get1 = ph == 0 ? 0x5210u : ph == 1 ? 0x6210u : 0x7410u;
        s.put0 = ph == 0 ? 0x1440u : ph == 1 ? 0x4404u : 0x4044u;
        s.put1 = ph == 0 ? 0x4244u : ph == 1 ? 0x2441u : 0x4414u;
        s.put2 = ph == 0 ? 0x4434u : ph == 1 ? 0x4344u : 0x3442u;
        s.mask0 = ph == 0 ? 0x03000003u : ph == 1 ? 0x00000300u : 0x00030000u;
        s.mask1 = ph == 0 ? 0x00030000u : ph == 1 ? 0x03000003u : 0x00000300u;
        s.mask2 = ph == 0 ? 0x00000300u : ph == 1 ? 0x00030000u : 0x03000003u;
    } else if (ch == 4) {
        s.get0 = ph | ((4u + ph) << 4);
        s.put0 = 0x4444u & ~(0xFu << (4 * ph));
        s.put1 = 4 * ph;
        s.mask0 = 3u << (8 * ph);
    }
    return s;
}

// The 16 plane bytes of a unit.
template <int CH>
__device__ __forceinline__ void get_unit(const uint32_t (&w)[4 * CH], const PlaneSel &s,
                                         uint32_t (&G)[4])
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if constexpr (CH == 1)
            G[q] = w[q];
        else if constexpr (CH == 3)
            G[q] = __byte_perm(__byte_perm(w[3 * q], w[3 * q + 1], s.get0), w[3 * q + 2], s.get1);
        else
            G[q] = __byte_perm(__byte_perm(w[4 * q], w[4 * q + 1], s.get0),
                               __byte_perm(w[4 * q + 2], w[4 * q + 3], s.get0), 0x5410u);
    }
}

// Pairs P (the low two bits of each byte; the others are ignored) into the
// plane bytes of a unit: per word one byte_perm and one masked merge.
template <int CH>
__device__ __forceinline__ void put_unit(uint32_t (&w)[4 * CH], const PlaneSel &s,
                                         const uint32_t (&P)[4])
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if constexpr (CH == 1) {
            w[q] = (w[q] & ~0x03030303u) | (P[q] & 0x03030303u);
        } else if constexpr (CH == 3) {
            w[3 * q] = (w[3 * q] & ~s.mask0) | (__byte_perm(P[q], 0u, s.put0) & s.mask0);
            w[3 * q + 1] = (w[3 * q + 1] & ~s.mask1) | (__byte_perm(P[q], 0u, s.put1) & s.mask1);
            w[3 * q + 2] = (w[3 * q + 2] & ~s.mask2) | (__byte_perm(P[q], 0u, s.put2) & s.mask2);
        } else {
#pragma unroll
            for (int t = 0; t < 4; ++t)
                w[4 * q + t] = (w[4 * q + t] & ~s.mask0) |
                               (__byte_perm(P[q], 0u, 0x1111u * t) & s.mask0);
        }
    }
}

// XOR of differences D (byte t%4 of word t/4 for plane byte t) into a unit's words.
template <int CH>
__device__ __forceinline__ void xor_unit(uint32_t (&w)[4 * CH], const PlaneSel &s,
                                         const uint32_t (&D)[4])
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if constexpr (CH == 1) {
            w[q] ^= D[q];
        } else if constexpr (CH == 3) {
            w[3 * q] ^= __byte_perm(D[q], 0u, s.put0);
            w[3 * q + 1] ^= __byte_perm(D[q], 0u, s.put1);
            w[3 * q + 2] ^= __byte_perm(D[q], 0u, s.put2);
        } else {
#pragma unroll
            for (int t = 0; t < 4; ++t)
                w[4 * q + t] ^= __byte_perm(D[q], 0u, s.put0 | (t << s.put1));
        }
    }
}

// 16-byte vectors' words v -> the 16*CH bytes that start d bytes into them (d
// < 16): the word offset d / 4 by a switch, which a warp takes together where
// its lanes share d, the byte offset by one byte_perm per word.
template <int CH, int QW>
__device__ __forceinline__ void join_words(const uint32_t (&v)[4 * CH + 4], uint32_t sel,
                                           uint32_t (&o)[4 * CH])
{
#pragma unroll
    for (int q = 0; q < 4 * CH; ++q)
        o[q] = __byte_perm(v[q + QW], v[q + QW + 1], sel);
}

template <int CH>
__device__ __forceinline__ void join_unit(const uint32_t (&v)[4 * CH + 4], uint32_t d,
                                          uint32_t (&o)[4 * CH])
{
    const uint32_t sel = 0x3210u + 0x1111u * (d & 3u);
    switch (d >> 2) {
    case 0: join_words<CH, 0>(v, sel, o); break;
    case 1: join_words<CH, 1>(v, sel, o); break;
    case 2: join_words<CH, 2>(v, sel, o); break;
    default: join_words<CH, 3>(v, sel, o); break;
    }
}

// Words 4q .. 4q + 3 of w from a vector, and back.
template <int N>
__device__ __forceinline__ void set_vec(uint32_t (&w)[N], int q, const uint4 &v)
{
    w[4 * q] = v.x;
    w[4 * q + 1] = v.y;
    w[4 * q + 2] = v.z;
    w[4 * q + 3] = v.w;
}

template <int N>
__device__ __forceinline__ uint4 get_vec(const uint32_t (&w)[N], int q)
{
    return make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
}

// How an image's bytes fall into units.  Units are counted from stego byte h
// on, a 128-byte boundary of the stego (16-byte in a small image) from which
// the cover's bytes can be read as whole vectors: unit k is stego bytes [h +
// 16*CH*k, h + 16*CH*(k + 1)).  As 16*CH bytes are 16 pixels, its plane bytes
// sit at unit bytes ph + t*CH, t = 0..15, for every k, and belong to pixels x0 +
// 16k + t: rows of any length and buffers at any address take the same byte
// positions.  A warp's vectors then start on a cache line: from a 16-byte
// boundary alone every warp writes two half sectors (8192x8192x3 in place:
// 87 us against 60).  The unit's cover bytes start d = (cover + h) mod 16
// bytes into an aligned vector.  The bytes before and after the units (fewer
// than 400 and 32*CH) are done one by one.
struct Flat {
    uint32_t h, d, ph, x0;
    uint64_t nunits;
    PlaneSel sel;
};

// The flat units of a cover; false when it holds none or has another channel
// count.
// `lead`: with three channels, h moved on by one or two boundaries so that ph =
// 0, for the kernels that take that position at compile time.
__host__ __device__ inline bool make_flat(const uint8_t *cover, const uint8_t *stego, uint64_t C,
                                          uint32_t ch, uint32_t plane, bool lead, Flat &f)
{
    if (!(ch == 1 || ch == 3 || ch == 4))
        return false;
    const uint32_t align = C >= 16384u ? 128u : 16u;
    f.h = (uint32_t)(-(uintptr_t)stego & (align - 1u));
    f.d = (uint32_t)(((uintptr_t)cover + f.h) & 15u);
    if (f.h < f.d)
        f.h += align; // the vector around the first cover byte would start before the cover
    while (lead && ch == 3u && f.h % 3u != plane)
        f.h += align;
    f.ph = (plane + 192u * ch - f.h % (3u * ch)) % ch;
    f.x0 = (f.h + f.ph - plane) / ch;
    f.nunits = 0;
    f.sel = make_sel(ch, f.ph);
    const uint64_t ub = 16u * ch;
    // one vector more than the units' own is read when d != 0
    const uint64_t need = f.h + (f.d ? 16u - f.d : 0u);
    if (C < need + ub)
        return false;
    f.nunits = (C - need) / ub;
    return true;
}

} // namespace stego

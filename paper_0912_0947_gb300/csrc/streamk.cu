// streamk.cu -- the stream layout with k = 1..4 bits per carrying byte, over
// every cover byte or over one colour plane in pixel order (Section VI step
// 2's "separate any one plane").  The variant space between the one-bit
// stream and the paper's two bits per byte (Section VI step 7c-f):
//
//   stream bit b  ->  bit (k - 1 - b mod k) of carrying byte b / k,
//   carrying byte x = cover byte x (all bytes) or x*channels + plane,
//
// S = BE32(8m) || msg (header) or msg.  When 8|S| is not a multiple of k, the
// last carrying byte changes only its top (8|S| mod k) field bits.  k = 1 over
// all bytes is handled by stream1.cu.
//
// Kernels:
//   embedk_units<K,STATS,FLAT>, embedk_units_async<K,CH,STATS,FLAT>  all bytes,
//       or one plane of 1, 3 or 4 channels: a unit of 16 carrying bytes (CH
//       vectors of the stego) carries 16K stream bits, assembled big-endian
//       into one 64-bit word and cut into 16 K-bit fields; out of place the
//       whole cover moves once, 2C + |S| bytes.  FLAT: buffers at any addresses
//       (units from the stego's 128-byte boundary on, see Flat; the stream cut
//       at any bit); else both 16-byte aligned, where unit u carries stream
//       bytes [2Ku, 2Ku + 2K).
//   embedk_bytes<STATS>  any alignment, any k, either carrying order: one
//       thread per carrying byte (other channel counts, one plane in place at
//       an odd address, covers of less than a few vectors; out of place with
//       one plane, after a copy of the cover).
//   extractk_units<K,CH,FLAT>  same layouts; FLAT: a stego at any address.
//   extractk_bytes  any alignment, any k, either carrying order.
// The header's 32 bits are read by warp 0 of each CTA: lane l loads stream
// bit l from its carrying byte and one ballot gathers them.
#include <cstring>

#include "async_copy.cuh"
#include "s1_device.cuh"
#include "unit_device.cuh"

namespace stego {
namespace {

// The installed launch shapes are tuned for the one-bit kernels; these
// kernels (other register counts) take as many resident CTAs as occupancy
// allows instead of a tuned CTA count.
constexpr int kAnyCtas = 0;

struct KView {
    const uint8_t *cover; // embed: cover; extract: stego
    uint8_t *stego;       // embed output
    const uint8_t *msg;   // embed message
    uint8_t *out;         // extract output
    uint64_t C;           // cover bytes
    uint64_t n_carry;     // carrying bytes processed (embed) / available (extract)
    uint64_t t_bits;      // embed: stream bits 8|S|
    uint64_t slen;        // embed: stream bytes
    uint64_t cap, raw_len;
    uint32_t k, header, nbits, plane_only;
    uint32_t channels, plane;
    stego_result *res;
    uint64_t res_msg_bytes;
    uint64_t full_units;  // embed: units wholly inside the stream, t_bits / 16k
    uint64_t part_units;  // embed: units touching the stream, ceil(t_bits / 16k)
    uint32_t msg_w4;      // embed: msg - (header bytes) is 4-byte aligned
    uint32_t msg_w2;      // embed: msg - (header bytes) is 2-byte aligned
    StatSlot *slot;       // embed: per-stream statistics slot or nullptr
    uint32_t kmul;        // embed: 1 << k (a multiplier the compiler cannot see)
    uint32_t pad;
    Flat f;               // the units (f.nunits: those embedded; extract: of a FLAT launch
                          // the whole vectors' units, from u_lo on)
    uint64_t edge_end;    // embed: end of the cover bytes processed
    uint64_t u_lo;        // extract, FLAT: first unit whose vectors lie in the stego
};

__device__ __forceinline__ uint64_t carry_pos(const KView &a, uint64_t x)
{
    return a.plane_only ? x * a.channels + a.plane : x;
}

__device__ __forceinline__ uint32_t sbyte(const KView &a, uint64_t q)
{
    if (q >= a.slen)
        return 0u;
    if (a.header) {
        if (q < 4)
            return (a.nbits >> (24u - 8u * (uint32_t)q)) & 0xFFu;
        return __ldg(a.msg + (q - 4));
    }
    return __ldg(a.msg + q);
}

// The k-bit field of carrying byte x and the mask of its bits that carry
// stream data (all k, the top few for the last byte, none past the stream).
__device__ __forceinline__ void field_of(const KView &a, uint64_t x, uint32_t &f, uint32_t &fm)
{
    const uint32_t k = a.k;
    const uint64_t b0 = x * k;
    if (b0 >= a.t_bits) {
        f = fm = 0u;
        return;
    }
    const uint64_t left = a.t_bits - b0;
    const uint32_t valid = left < k ? (uint32_t)left : k;
    const uint32_t w = (sbyte(a, b0 >> 3) << 8) | sbyte(a, (b0 >> 3) + 1);
    const uint32_t off = (uint32_t)(b0 & 7u);
    f = (w >> (16u - off - k)) & ((1u << k) - 1u);
    fm = ((1u << valid) - 1u) << (k - valid);
}

__device__ __forceinline__ void embed_res(const KView &a, bool stats)
{
    if (a.res && blockIdx.x == 0 && threadIdx.x == 0) {
        a.res->msg_bytes = a.res_msg_bytes;
        a.res->status = STEGO_OK;
        a.res->reserved = 0;
        if (!stats) {
            a.res->changed = 0;
            a.res->sse = 0;
        }
    }
}

// The one vector where the stream ends, field by field (a call of its own
// keeps the hot loop's registers low).
__device__ __noinline__ uint4 stream_end_vector(const KView &a, uint64_t x, uint4 c)
{
    uint32_t ow[4] = {c.x, c.y, c.z, c.w};
    for (int t = 0; t < 16; ++t) {
        uint32_t fv, fm;
        field_of(a, x + t, fv, fm);
        const uint32_t s = 8 * (t & 3);
        ow[t >> 2] = (ow[t >> 2] & ~(fm << s)) | ((fv & fm) << s);
    }
    return make_uint4(ow[0], ow[1], ow[2], ow[3]);
}

// Stream bytes [2Kv, 2Kv + 2K) as a big-endian 64-bit word (whole vector
// inside the stream): word loads when they are message bytes on a 4-byte
// boundary, byte loads otherwise.  K = 3 packs its 6 bytes as two 24-bit
// halves instead, bytes 0-2 in the high word and 3-5 in the low one, each
// first byte on top (the form unit_fields<3> spreads).
template <int K>
__device__ __forceinline__ uint64_t stream_window(const KView &a, uint64_t v)
{
    uint64_t X = 0;
    const uint64_t q0 = 2u * K * v;
    const uint64_t hb = a.header ? 4u : 0u;
    const uint8_t *mp = a.msg + (q0 - hb);
    // q0 is a multiple of 4 for even K (of 2 for K = 3), so mp's alignment
    // is the launch's
    if constexpr (K == 3) {
        uint32_t v01, v23;
        if (q0 >= hb && a.msg_w2) {
            const unsigned short *hp = reinterpret_cast<const unsigned short *>(mp);
            const uint32_t h0 = __ldg(hp), h1 = __ldg(hp + 1), h2 = __ldg(hp + 2);
            v01 = __byte_perm(h0, h1, 0x2014u); // bytes 0, 1, 2 from the top; byte 3 zero
            v23 = __byte_perm(h1, h2, 0x2145u); // bytes 3, 4, 5
        } else {
            v01 = (sbyte(a, q0) << 16) | (sbyte(a, q0 + 1) << 8) | sbyte(a, q0 + 2);
            v23 = (sbyte(a, q0 + 3) << 16) | (sbyte(a, q0 + 4) << 8) | sbyte(a, q0 + 5);
        }
        return ((uint64_t)v01 << 32) | v23;
    } else if ((K & 1) == 0 && q0 >= hb && a.msg_w4) {
#pragma unroll
        for (int i = 0; i < K / 2; ++i) {
            const uint32_t w = __ldg(reinterpret_cast<const uint32_t *>(mp) + i);
            X |= (uint64_t)__byte_perm(w, 0u, 0x0123u) << (32 - 32 * i);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 2 * K; ++i)
            X |= (uint64_t)sbyte(a, q0 + i) << (56 - 8 * i);
    }
    return X;
}

// The 16K stream bits of the carrying bytes x .. x + 15 for any x, in
// stream_window's form: the aligned message words around the 2K or 2K + 1
// stream bytes that hold them, byte-shifted, reversed and cut at bit K*x % 8;
// byte by byte where those words are not all inside the message.
template <int K>
__device__ __forceinline__ uint64_t stream_window_at(const KView &a, uint64_t x)
{
    constexpr int NW = K >= 3 ? 3 : 2; // words that hold 3 + 2K + 1 bytes
    const uint64_t b0 = x * K, q = b0 >> 3;
    const uint32_t s = (uint32_t)(b0 & 7u);
    const uint64_t hb = a.header ? 4u : 0u;
    const uintptr_t p = (uintptr_t)a.msg + (uintptr_t)(q - hb);
    const uint32_t al = (uint32_t)(p & 3u);
    uint32_t hi, lo, more; // stream bytes q .. q + 3, q + 4 .. q + 7 (first on top), q + 8
    if (q >= hb + al && q - hb - al + 4u * NW <= a.slen - hb) {
        const uint32_t *w = reinterpret_cast<const uint32_t *>(p - al);
        uint32_t v[3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
            v[i] = i < NW ? __ldg(w + i) : 0u;
        hi = __byte_perm(__funnelshift_r(v[0], v[1], 8 * al), 0u, 0x0123u);
        lo = __byte_perm(__funnelshift_r(v[1], v[2], 8 * al), 0u, 0x0123u);
        more = v[2] >> (8 * al);
    } else {
        hi = lo = more = 0u;
#pragma unroll 1
        for (int i = 0; i < 9; ++i) { // shifted in from below
            hi = __funnelshift_l(lo, hi, 8);
            lo = __funnelshift_l(more << 24, lo, 8);
            more = i < 2 * K + 1 ? sbyte(a, q + i) : 0u;
        }
    }
    const uint32_t h = __funnelshift_l(lo, hi, s), l = __funnelshift_l(more << 24, lo, s);
    if constexpr (K == 3)
        return ((uint64_t)(h >> 8) << 32) | ((h & 0xFFu) << 16) | (l >> 16);
    else if constexpr (K == 4)
        return ((uint64_t)h << 32) | l;
    else
        return (uint64_t)h << 32;
}

// A unit is 16 consecutive carrying bytes: 16 consecutive cover bytes (all
// bytes, CH = 1) or the plane bytes of 16 consecutive pixels (CH = 3 or 4
// channels), i.e. CH 16-byte vectors.  Its 16 carrying bytes are gathered into
// one 16-byte value, transformed as one vector of the all-bytes layout, and
// the change is XORed back.
template <int CH>
__device__ __forceinline__ void load_unit(const uint8_t *base, uint64_t u, uint32_t (&w)[4 * CH])
{
    const uint4 *p = reinterpret_cast<const uint4 *>(base) + u * CH;
#pragma unroll
    for (int j = 0; j < CH; ++j)
        set_vec(w, j, __ldcs(p + j));
}

// Word i (carrying bytes 4i..4i+3, field in each byte's low K bits) of a
// unit whose stream window is X (stream bytes big-endian, the first in bits
// 56..63; for K = 3 two 24-bit halves).  K = 1, 4 fill the four byte lanes
// from replicated stream bytes with fixed per-lane shifts, K = 2 with one
// multiply; K = 3 (fields across byte boundaries) takes the word's 12 bits
// t and multiplies by 2^24 + 4: the two copies of t do not overlap, and
// leave fields 1, 3 at bits 8, 24 and fields 0, 2 at bits 11, 27, which one
// shift by 11 brings to bits 0, 16.
template <int K>
__device__ __forceinline__ uint32_t unit_fields(uint64_t X, int i)
{
    const uint32_t hi = (uint32_t)(X >> 32), lo = (uint32_t)X;
    if constexpr (K == 1) {
        // stream byte i/2; even words take its bits 7..4, odd words 3..0
        const uint32_t r = __byte_perm(hi, 0u, i < 2 ? 0x3333u : 0x2222u);
        return (i & 1) ? s1::spread_lo(r) : s1::spread_hi(r);
    } else if constexpr (K == 2) {
        // stream byte i; lane l takes its bits 7-2l and 6-2l: the products
        // b << 10l occupy disjoint bit ranges, and bits 8l+6, 8l+7 of their
        // sum hold pair l (b's bits 7-2l, 6-2l)
        const uint32_t b = __byte_perm(hi, 0u, 0x4440u | (3 - i)); // (hi >> (24 - 8i)) & 0xFF
        return ((b * 0x40100401u) >> 6) & 0x03030303u;
    } else if constexpr (K == 4) {
        // stream bytes 2i, 2i+1; lanes take high nibble, low nibble, high, low
        const uint32_t r = __byte_perm(i < 2 ? hi : lo, 0u, (i & 1) ? 0x0011u : 0x2233u);
        return ((r >> 4) & 0x000F000Fu) | (r & 0x0F000F00u);
    } else {
        static_assert(K == 3, "one to four bits per byte");
        const uint32_t h = i < 2 ? hi : lo;
        const uint32_t t = (i & 1) ? (h & 0xFFFu) : (h >> 12);
        const uint32_t p = t * 0x01000004u;
        return (p & 0x07000700u) | ((p & 0x38003800u) >> 11);
    }
}

// The inverse: a unit's stream window from its 16 carrying bytes g (words
// of four), fields in the low K bits.  K = 1 and 2 gather the four lanes of
// a word with one multiply (the partial products of the wanted bits land in
// disjoint bit ranges of the top byte, all others below it or past bit 31);
// K = 4 joins nibble pairs.
template <int K>
__device__ __forceinline__ uint64_t unit_window(const uint32_t (&g)[4])
{
    if constexpr (K == 1) {
        const uint32_t b0 = (s1::gather4(g[0]) << 4) | s1::gather4(g[1]);
        const uint32_t b1 = (s1::gather4(g[2]) << 4) | s1::gather4(g[3]);
        return (uint64_t)((b0 << 24) | (b1 << 16)) << 32;
    } else if constexpr (K == 2) {
        uint32_t hi = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) // lane l -> bits 30-2l, 31-2l of the product
            hi |= (((g[i] & 0x03030303u) * 0x40100401u) >> 24) << (24 - 8 * i);
        return (uint64_t)hi << 32;
    } else {
        static_assert(K == 4, "k = 3: unit_window3");
        uint32_t b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t m = g[i] & 0x0F0F0F0Fu;
            b[i] = ((m << 4) | (m >> 8)) & 0x00FF00FFu; // bytes 2i (lane 0), 2i+1 (lane 2)
        }
        const uint32_t hi = __byte_perm(b[0], b[1], 0x0246u); // b0.l0 b0.l2 b1.l0 b1.l2, first on top
        const uint32_t lo = __byte_perm(b[2], b[3], 0x0246u);
        return ((uint64_t)hi << 32) | lo;
    }
}

// k = 3: the unit's 48 stream bits as two 24-bit halves (words 0-1, 2-3),
// first bit on top.  Per word, one multiply by 2^11 + 1 joins the fields of
// bytes 0, 1 into bits 8-13 and those of bytes 2, 3 into bits 24-29 (the
// shifted copies do not overlap, so nothing carries); the high half of a
// second product, by 2^30 + 2^8, puts the first pair above the second at
// bits 0-11, with a copy of the second pair at bits 22-27 that the 12-bit
// shift of the first word pushes out and a mask of the second word drops.
// The multiplies run on the FMA pipe, which the k = 3 gather left idle.
__device__ __forceinline__ void unit_window3(const uint32_t (&g)[4], uint32_t &v01, uint32_t &v23)
{
    uint32_t t[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        t[i] = __umulhi(((g[i] & 0x07070707u) * 0x801u) & 0x3F003F00u, 0x40000100u);
    v01 = (t[0] << 12) | (t[1] & 0xFFFu);
    v23 = (t[2] << 12) | (t[3] & 0xFFFu);
}

// Units each thread of an extract keeps in flight per loop iteration.  A plane
// unit is already CH vectors; all-bytes units are single vectors, of which the
// extract batches four (measured on the 201 MB cover, k = 2: 43.0 us
// against 45.1 us with one, while one is fastest for the embed: 101.4 us
// against 114.7 us with two and 148.5 us with four).
constexpr int kExtractAllBytesUnits = 4;
template <int CH>
__host__ __device__ constexpr int units_per_iter()
{
    return CH == 1 ? kExtractAllBytesUnits : 1;
}

// Bytes outside the units, [0, f.h) and [f.h + 16*CH*nunits, edge_end), by the
// calling CTA: plane bytes take their field, the other bytes of those pixels
// are copied (in place only what changes is written).
template <int CH, bool STATS>
__device__ __forceinline__ void embedk_edges(const KView &a, unsigned long long &changed,
                                             unsigned long long &sse)
{
    const uint64_t t0 = a.f.h + 16u * CH * a.f.nunits;
    const uint32_t nt = a.edge_end > t0 ? (uint32_t)(a.edge_end - t0) : 0u;
    for (uint32_t e = threadIdx.x; e < a.f.h + nt; e += blockDim.x) {
        const uint64_t k = e < a.f.h ? e : t0 + (e - a.f.h);
        const uint32_t cb = a.cover[k];
        uint32_t ob = cb;
        if (k % CH == a.plane) {
            uint32_t fv, fm;
            field_of(a, k / CH, fv, fm);
            ob = (cb & ~fm) | (fv & fm);
        }
        if (ob != cb || a.stego != a.cover)
            a.stego[k] = (uint8_t)ob;
        if (STATS) {
            const uint32_t dd = ob > cb ? ob - cb : cb - ob;
            changed += dd != 0;
            sse += dd * dd;
        }
    }
}

// The 16 carrying bytes c of unit u (first carrying byte x) -> o, its stream
// window X read when the unit lies wholly inside the stream.
template <int K>
__device__ __forceinline__ void embed_fields(const KView &a, uint64_t u, uint64_t x, uint64_t X,
                                             const uint32_t (&c)[4], uint32_t (&o)[4])
{
    constexpr uint32_t BYTEMASK = ((1u << K) - 1u) * 0x01010101u;
    if (u < a.full_units) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            o[i] = (c[i] & ~BYTEMASK) | unit_fields<K>(X, i);
    } else {
        const uint4 e = stream_end_vector(a, x, make_uint4(c[0], c[1], c[2], c[3]));
        o[0] = e.x;
        o[1] = e.y;
        o[2] = e.z;
        o[3] = e.w;
    }
}

// Embed over all-bytes units, single vectors, one per thread and iteration
// (see kExtractAllBytesUnits).  Units wholly past the stream are copied.  FLAT:
// a cover at another address mod 16 than the stego is read as the two vectors
// around the unit's bytes (the second is the neighbour's first: an L1 hit).
// All bytes at k = 2, 3, 4 are bound by instructions as much as by HBM (ALU pipe
// 60% at k = 2; 8192x8192x3 77.1 / 84.6 / 83.4 us).  Buffers at odd addresses
// ran one thread per carrying byte before: 5471x3647x3, cover 13 bytes past a
// boundary, k = 2, 3, 4: 220 / 215 / 217 -> 31.3 / 34.3 / 34.5 us, both 13 bytes
// past, k = 2: 220 -> 27.5.  An odd message with aligned covers (byte loads
// before) 28.8 -> 26.8.
template <int K, bool STATS, bool FLAT>
__global__ void __launch_bounds__(512, K >= 3 ? 3 : 0) embedk_units(KView a)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    unsigned long long changed = 0, sse = 0;
    embed_res(a, STATS);
    if (blockIdx.x == gridDim.x - 1) // the CTA with the fewest units
        embedk_edges<1, STATS>(a, changed, sse);
    const uint64_t nunits = a.f.nunits;
    const uint4 *__restrict__ src =
        reinterpret_cast<const uint4 *>(a.cover + (FLAT ? a.f.h - a.f.d : 0u));
    uint4 *dst = reinterpret_cast<uint4 *>(a.stego + (FLAT ? a.f.h : 0u));
    for (uint64_t u = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nunits;
         u += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t w[4];
        if (FLAT && a.f.d) {
            uint32_t v[8];
            set_vec(v, 0, __ldcs(src + u));
            set_vec(v, 1, __ldcs(src + u + 1));
            join_unit<1>(v, a.f.d, w);
        } else {
            set_vec(w, 0, __ldcs(src + u));
        }
        if (u < a.part_units) {
            const uint64_t x = (FLAT ? a.f.x0 : 0u) + 16u * u;
            uint64_t X = 0;
            if (u < a.full_units)
                X = FLAT ? stream_window_at<K>(a, x) : stream_window<K>(a, u);
            uint32_t o[4], d[4];
            embed_fields<K>(a, u, x, X, w, o);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                d[i] = o[i] ^ w[i];
            if (STATS)
                unit_stats<K>(o, w, d, a.kmul, changed, sse);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                w[i] = o[i];
        }
        __stcs(dst + u, get_vec(w, 0));
    }
    if (STATS)
        block_stats(changed, sse, a.res, a.slot);
}

// Plane units (CH = 3 or 4) with a two-stage copy pipeline per warp: while
// the warp embeds the units of one iteration from shared memory, the cover
// vectors of its next iteration are on their way there (cp.async, memory
// order, coalesced: a lane's own unit is 16*CH bytes from its neighbour's)
// and the next units' stream windows on their way to registers.  Each lane
// then takes its unit from shared memory, embeds it as embedk_units does and
// writes it back; the warp stores its vectors in memory order.  FLAT with
// cover and stego at different addresses mod 16: the stage holds the 32*CH + 1
// aligned cover vectors around the warp's bytes, of which each lane reads CH +
// 1.  CTAs of at most kAsyncThreads threads (the staging area holds that many
// warps).  HBM-bound: k = 2, plane 0 of 8192x8192x3 67.5 us; with the plane's
// position at run time (one kernel for all) as fast as at compile time (68.9).
// 3839x2159x3 in packed stacks, k = 3, plane 1 (a copy and a kernel of one
// thread per carrying byte before): 39.2 -> 14.4 us.
constexpr int kAsyncThreads = 256;
template <int K, int CH, bool STATS, bool FLAT>
__global__ void __launch_bounds__(kAsyncThreads) embedk_units_async(KView a)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    static_assert(CH > 1, "plane units only");
    constexpr uint32_t SV = unit_stage_slots<CH>() + (FLAT ? 1u : 0u);
    __shared__ uint4 stage[(kAsyncThreads / 32) * 2 * SV];
    uint4 *const sw = stage + (threadIdx.x >> 5) * 2 * SV;
    const uint32_t lane = threadIdx.x & 31u;
    unsigned long long changed = 0, sse = 0;
    embed_res(a, STATS);
    if (blockIdx.x == gridDim.x - 1) // the CTA with the fewest units
        embedk_edges<CH, STATS>(a, changed, sse);
    const uint64_t nunits = a.f.nunits;
    const bool joined = FLAT && a.f.d;
    const uint64_t vend = nunits * CH;              // vectors written
    const uint64_t vread = vend + (joined ? 1u : 0u); // and read
    const uint4 *__restrict__ cv =
        reinterpret_cast<const uint4 *>(a.cover + (FLAT ? a.f.h - a.f.d : 0u));
    uint4 *const ov = reinterpret_cast<uint4 *>(a.stego + (FLAT ? a.f.h : 0u));
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    auto issue = [&](uint64_t ub, uint32_t s) { // the warp's vectors from unit ub -> stage s
        const uint64_t v0 = ub * CH;
#pragma unroll
        for (int j = 0; j < CH; ++j)
            if (v0 + 32u * j + lane < vread)
                cp_async16(sw + s * SV + unit_stage_slot<CH>(32u * j + lane), cv + v0 + 32u * j + lane);
        if (FLAT && lane == 0 && v0 + 32u * CH < vread)
            cp_async16(sw + s * SV + unit_stage_slot<CH>(32u * CH), cv + v0 + 32u * CH);
        cp_async_commit();
    };
    auto window = [&](uint64_t u) {
        if (u >= nunits || u >= a.full_units)
            return (uint64_t)0;
        return FLAT ? stream_window_at<K>(a, a.f.x0 + 16u * u) : stream_window<K>(a, u);
    };
    uint64_t u = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; // u - lane: the same for the warp
    if (u - lane < nunits) {
        issue(u - lane, 0);
        uint64_t X = window(u);
        uint32_t s = 0;
        for (;;) {
            const uint64_t un = u + step;
            const bool next = un - lane < nunits;
            uint64_t Xn = 0;
            if (next) {
                issue(un - lane, s ^ 1u);
                Xn = window(un);
                cp_async_wait<1>(); // this iteration's copies landed (the next may be pending)
            } else {
                cp_async_wait<0>();
            }
            __syncwarp(); // every lane's copies visible to the warp
            uint4 *const st = sw + s * SV;
            const bool embeds = u < nunits && u < a.part_units;
            if (joined || embeds) {
                uint32_t w[4 * CH];
                if (joined) {
                    uint32_t v[4 * CH + 4];
#pragma unroll
                    for (int q = 0; q <= CH; ++q)
                        set_vec(v, q, st[unit_stage_slot<CH>(CH * lane + q)]);
                    join_unit<CH>(v, a.f.d, w);
                    __syncwarp(); // the neighbour has read this lane's first vector
                } else {
#pragma unroll
                    for (int q = 0; q < CH; ++q)
                        set_vec(w, q, st[unit_stage_slot<CH>(CH * lane + q)]);
                }
                if (embeds) {
                    uint32_t c[4], o[4], d[4];
                    get_unit<CH>(w, a.f.sel, c);
                    embed_fields<K>(a, u, (FLAT ? a.f.x0 : 0u) + 16u * u, X, c, o);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        d[i] = o[i] ^ c[i];
                    if (STATS)
                        unit_stats<K>(o, c, d, a.kmul, changed, sse);
                    xor_unit<CH>(w, a.f.sel, d);
                }
#pragma unroll
                for (int q = 0; q < CH; ++q)
                    st[unit_stage_slot<CH>(CH * lane + q)] = get_vec(w, q);
            }
            __syncwarp(); // the rewritten units visible to the storing lanes
            const uint64_t v0 = (u - lane) * CH;
#pragma unroll
            for (int j = 0; j < CH; ++j)
                if (v0 + 32u * j + lane < vend)
                    __stcs(ov + v0 + 32u * j + lane, st[unit_stage_slot<CH>(32u * j + lane)]);
            if (!next)
                break;
            // stage s is refilled two iterations on, after every lane passed
            // the barriers above and read its own memory-order slots
            X = Xn;
            u = un;
            s ^= 1u;
        }
    }
    if (STATS)
        block_stats(changed, sse, a.res, a.slot);
}

// One thread per carrying byte x < n_carry (all bytes: the bytes past the
// stream are copied; one plane: only plane bytes are written).
template <bool STATS>
__global__ void __launch_bounds__(512) embedk_bytes(KView a)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    unsigned long long changed = 0, sse = 0;
    embed_res(a, STATS);
    for (uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; x < a.n_carry;
         x += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t fv, fm;
        field_of(a, x, fv, fm);
        const uint64_t p = carry_pos(a, x);
        const uint32_t cb = a.cover[p]; // plain load: cover may equal stego
        const uint32_t ob = (cb & ~fm) | (fv & fm);
        a.stego[p] = (uint8_t)ob;
        if (STATS) {
            const uint32_t d = ob > cb ? ob - cb : cb - ob;
            changed += d != 0;
            sse += d * d;
        }
    }
    if (STATS)
        block_stats(changed, sse, a.res, a.slot);
}

// Stream bit b read back from the stego.
__device__ __forceinline__ uint32_t stream_bit(const KView &a, uint64_t b)
{
    const uint64_t x = b / a.k;
    const uint32_t pos = a.k - 1u - (uint32_t)(b - x * a.k);
    return (a.cover[carry_pos(a, x)] >> pos) & 1u;
}

// Length, status and first message bit of an extraction; block 0 publishes
// the result.  With the header, warp 0 reads stream bits 0..31 (one per lane)
// and one ballot assembles the count.
__device__ __forceinline__ int extractk_prologue(const KView &a, uint64_t &len)
{
    __shared__ int s_status;
    __shared__ unsigned long long s_len;
    const uint64_t avail = a.n_carry * a.k; // stream bits the stego holds
    if (a.header) {
        if (threadIdx.x < 32) {
            const uint32_t l = threadIdx.x;
            const uint32_t bit = (l < avail) ? stream_bit(a, l) : 0u;
            const uint32_t nbits = __brev(__ballot_sync(0xFFFFFFFFu, bit));
            if (l == 0) {
                int st = STEGO_OK;
                if (avail < 32u || (nbits & 7u) || 32ull + nbits > avail)
                    st = STEGO_E_BAD_HEADER;
                else if ((uint64_t)(nbits >> 3) > a.cap)
                    st = STEGO_E_MSG_TOO_SMALL;
                s_status = st;
                s_len = st == STEGO_OK ? (nbits >> 3) : 0u;
            }
        }
    } else if (threadIdx.x == 0) {
        s_status = STEGO_OK;
        s_len = a.raw_len;
    }
    __syncthreads();
    len = s_len;
    const int status = s_status;
    if (a.res && blockIdx.x == 0 && threadIdx.x == 0) {
        a.res->changed = 0;
        a.res->sse = 0;
        a.res->msg_bytes = len;
        a.res->status = status;
        a.res->reserved = 0;
    }
    return status;
}

// Unit u's words: its vectors, or (FLAT) its bytes from the vectors around them.
template <int CH, bool FLAT>
__device__ __forceinline__ void read_unit(const KView &a, uint64_t u, uint32_t (&w)[4 * CH])
{
    if constexpr (FLAT) {
        const uint4 *p = reinterpret_cast<const uint4 *>(a.cover - a.f.d) + u * CH;
        uint32_t v[4 * CH + 4];
#pragma unroll
        for (int j = 0; j <= CH; ++j)
            set_vec(v, j, __ldg(p + j));
        join_unit<CH>(v, a.f.d, w);
    } else {
        load_unit<CH>(a.cover, u, w);
    }
}

// k = 3 units of the extract: unit u yields the 6 stream bytes [6u, 6u + 6),
// so a lane pair (units 2j, 2j + 1) holds 12 consecutive message bytes and
// writes them as three aligned words: the even lane its first four bytes
// and its last two joined to the odd lane's first two (one shuffle), the
// odd lane its last four.  The loop runs while the warp's first unit is in
// range, so every lane reaches the shuffle; pairs at the header, at the
// message's end or on an unaligned output store 16-bit halves or bytes.
template <int CH, bool FLAT>
__device__ __forceinline__ void extract3_units(const KView &a, uint64_t ulo, uint64_t nunits,
                                               uint64_t hb, uint64_t sbytes)
{
    constexpr int U = units_per_iter<CH>();
    const uint32_t lane = threadIdx.x & 31u;
    const bool odd = (lane & 1u) != 0;
    // stream byte 12j lands at out + 12j - hb: word-aligned for every j or none
    const bool words = (((uintptr_t)a.out - hb) & 3u) == 0;
    for (uint64_t u0 = (uint64_t)blockIdx.x * blockDim.x * U + threadIdx.x; u0 - lane < nunits;
         u0 += (uint64_t)gridDim.x * blockDim.x * U) {
        uint32_t w[U][4 * CH];
#pragma unroll
        for (int r = 0; r < U; ++r) {
            const uint64_t u = u0 + (uint64_t)r * blockDim.x;
            if (u < nunits && (!FLAT || u >= ulo)) {
                read_unit<CH, FLAT>(a, u, w[r]);
            } else {
#pragma unroll
                for (int j = 0; j < 4 * CH; ++j)
                    w[r][j] = 0;
            }
        }
#pragma unroll
        for (int r = 0; r < U; ++r) {
            const uint64_t u = u0 + (uint64_t)r * blockDim.x;
            uint32_t g[4], v01, v23;
            get_unit<CH>(w[r], a.f.sel, g);
            unit_window3(g, v01, v23);
            const uint32_t P = __byte_perm(v01, v23, 0x6012u); // stream bytes 0-3, memory order
            const uint32_t Q = __byte_perm(v23, 0u, 0x4401u);  // stream bytes 4-5
            const uint32_t Pn = __shfl_down_sync(0xFFFFFFFFu, P, 1);
            const uint64_t q2 = 6u * (u & ~1ull); // first stream byte of the pair
            if (words && (u | 1u) < nunits && (u & ~1ull) >= ulo && q2 >= hb && q2 + 12 <= sbytes) {
                uint32_t *op = reinterpret_cast<uint32_t *>(a.out + (q2 - hb));
                if (odd) {
                    op[2] = __byte_perm(P, Q, 0x5432u);
                } else {
                    op[0] = P;
                    op[1] = __byte_perm(Q, Pn, 0x5410u);
                }
            } else if (u < nunits && (!FLAT || u >= ulo)) {
                const uint64_t q0 = 6u * u; // first stream byte of the unit
                if (q0 >= hb && q0 + 6 <= sbytes && ((q0 - hb + (uintptr_t)a.out) & 1u) == 0) {
                    unsigned short *op = reinterpret_cast<unsigned short *>(a.out + (q0 - hb));
                    op[0] = (unsigned short)P;
                    op[1] = (unsigned short)(P >> 16);
                    op[2] = (unsigned short)Q;
                } else {
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        const uint64_t q = q0 + i;
                        if (q >= hb && q < sbytes)
                            a.out[q - hb] = (uint8_t)(i < 3 ? v01 >> (16 - 8 * i) : v23 >> (40 - 8 * i));
                    }
                }
            }
        }
    }
}

// Extract over units: unit u yields stream bytes [2Ku, 2Ku + 2K); U units per
// thread per iteration, loads first.  FLAT: a stego at any address, its units
// read as the CH + 1 aligned vectors around them (3839x2159x3, k = 3, plane 1:
// 16.6 us bit by bit -> 5.5; 5471x3647x3, all bytes, k = 2, 3: 71 / 104 -> 17.3 /
// 20.5).  Stream bytes before the
// first and past the last unit whose vectors lie in the stego go bit by bit.
template <int K, int CH, bool FLAT>
__global__ void __launch_bounds__(512) extractk_units(KView a)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    uint64_t len;
    if (extractk_prologue(a, len) != STEGO_OK)
        return;
    const uint64_t hb = a.header ? 4u : 0u;       // stream bytes before the message
    const uint64_t sbytes = len + hb;              // stream bytes to recover
    const uint64_t want = (sbytes + 2 * K - 1) / (2 * K);
    const uint64_t nunits = want < a.f.nunits ? want : a.f.nunits;
    const uint64_t ulo = FLAT ? (a.u_lo < nunits ? a.u_lo : nunits) : 0u;
    // stream bytes [u0, u1) are the units'; the others one by one
    const uint64_t u1 = 2u * K * nunits < sbytes ? 2u * K * nunits : sbytes;
    const uint64_t u0 = 2u * K * ulo < u1 ? 2u * K * ulo : u1;
    for (uint64_t qq = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; qq < sbytes - (u1 - u0);
         qq += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t q = qq < u0 ? qq : qq + (u1 - u0);
        if (q < hb)
            continue;
        uint32_t v = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            v |= stream_bit(a, 8u * q + i) << (7 - i);
        a.out[q - hb] = (uint8_t)v;
    }
    if constexpr (K == 3) {
        extract3_units<CH, FLAT>(a, ulo, nunits, hb, sbytes);
    } else {
        constexpr int U = units_per_iter<CH>();
        for (uint64_t v0 = (uint64_t)blockIdx.x * blockDim.x * U + threadIdx.x; v0 < nunits;
             v0 += (uint64_t)gridDim.x * blockDim.x * U) {
            uint32_t w[U][4 * CH];
#pragma unroll
            for (int r = 0; r < U; ++r) {
                const uint64_t u = v0 + (uint64_t)r * blockDim.x;
                if (u < nunits && (!FLAT || u >= ulo))
                    read_unit<CH, FLAT>(a, u, w[r]);
            }
#pragma unroll
            for (int r = 0; r < U; ++r) {
                const uint64_t u = v0 + (uint64_t)r * blockDim.x;
                if (u >= nunits || (FLAT && u < ulo))
                    continue;
                uint32_t g[4];
                get_unit<CH>(w[r], a.f.sel, g);
                const uint64_t X = unit_window<K>(g);
                const uint64_t q0 = 2u * K * u; // first stream byte of the unit
                uint8_t *op = a.out + (q0 - hb);
                if ((K & 1) == 0 && q0 >= hb && q0 + 2 * K <= sbytes &&
                    (((uintptr_t)op & 3u) == 0)) {
                    // message bytes only, 4-byte aligned: K/2 word stores
#pragma unroll
                    for (int i = 0; i < K / 2; ++i)
                        reinterpret_cast<uint32_t *>(op)[i] =
                            __byte_perm((uint32_t)(X >> (32 - 32 * i)), 0u, 0x0123u);
                } else {
#pragma unroll
                    for (int i = 0; i < 2 * K; ++i) {
                        const uint64_t q = q0 + i; // stream byte
                        if (q >= hb && q < sbytes)
                            a.out[q - hb] = (uint8_t)(X >> (56 - 8 * i));
                    }
                }
            }
        }
    }
}

// Any alignment, any k, either carrying order: one thread per message byte.
__global__ void __launch_bounds__(512) extractk_bytes(KView a)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    uint64_t len;
    if (extractk_prologue(a, len) != STEGO_OK)
        return;
    const uint64_t first = a.header ? 32u : 0u;
    for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s < len;
         s += (uint64_t)gridDim.x * blockDim.x) {
        // walk the message byte's eight stream bits field by field: one
        // division per byte, one load per carrying byte touched
        const uint64_t b0 = first + 8u * s;
        uint64_t x = b0 / a.k;
        uint32_t r = (uint32_t)(b0 - x * a.k);
        uint32_t cb = a.cover[carry_pos(a, x)];
        uint32_t v = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            v |= ((cb >> (a.k - 1u - r)) & 1u) << (7 - i);
            if (++r == a.k && i < 7) {
                r = 0;
                cb = a.cover[carry_pos(a, ++x)];
            }
        }
        a.out[s] = (uint8_t)v;
    }
}

bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// Unit kernels exist for 1, 3 and 4 channels.
bool unit_layout(bool plane_only, const stego_geom *g)
{
    return !plane_only || g->channels == 1 || g->channels == 3 || g->channels == 4;
}

template <int K, bool STATS, bool FLAT>
const void *embed_units_for(uint32_t ch)
{
    switch (ch) {
    case 1: return (const void *)embedk_units<K, STATS, FLAT>;
    case 3: return (const void *)embedk_units_async<K, 3, STATS, FLAT>;
    default: return (const void *)embedk_units_async<K, 4, STATS, FLAT>;
    }
}

template <bool STATS, bool FLAT>
const void *embed_units_kernel(uint32_t k, uint32_t ch)
{
    switch (k) {
    case 1: return embed_units_for<1, STATS, FLAT>(ch);
    case 2: return embed_units_for<2, STATS, FLAT>(ch);
    case 3: return embed_units_for<3, STATS, FLAT>(ch);
    default: return embed_units_for<4, STATS, FLAT>(ch);
    }
}

template <int K, bool FLAT>
const void *extract_units_for(uint32_t ch)
{
    switch (ch) {
    case 1: return (const void *)extractk_units<K, 1, FLAT>;
    case 3: return (const void *)extractk_units<K, 3, FLAT>;
    default: return (const void *)extractk_units<K, 4, FLAT>;
    }
}

template <bool FLAT>
const void *extract_units_kernel(uint32_t k, uint32_t ch)
{
    switch (k) {
    case 1: return extract_units_for<1, FLAT>(ch);
    case 2: return extract_units_for<2, FLAT>(ch);
    case 3: return extract_units_for<3, FLAT>(ch);
    default: return extract_units_for<4, FLAT>(ch);
    }
}

} // namespace

cudaError_t sk_embed(const uint8_t *cover, uint8_t *stego, uint64_t C, uint32_t k, bool plane_only,
                     const stego_geom *g, const uint8_t *msg, uint64_t m, bool header,
                     bool stats, stego_result *res, const Shape &sh, cudaStream_t s,
                     StatSlot *slot)
{
    KView a;
    std::memset(&a, 0, sizeof(a));
    a.cover = cover;
    a.stego = stego;
    a.msg = msg;
    a.C = C;
    a.slen = m + (header ? 4u : 0u);
    a.t_bits = 8u * a.slen;
    a.k = k;
    a.header = header ? 1u : 0u;
    a.nbits = (uint32_t)(8u * m);
    a.plane_only = plane_only ? 1u : 0u;
    a.channels = plane_only ? g->channels : 1u;
    a.plane = plane_only ? g->plane : 0u;
    a.res = res;
    a.res_msg_bytes = m;
    a.slot = stats ? slot : nullptr;
    a.msg_w4 = (((uintptr_t)msg - (header ? 4u : 0u)) & 3u) == 0;
    a.msg_w2 = (((uintptr_t)msg - (header ? 4u : 0u)) & 1u) == 0;
    a.kmul = 1u << k;
    const bool inplace = cover == stego;
    const uint64_t t_carry = (a.t_bits + k - 1) / k; // carrying bytes the stream uses
    const int T = sh.threads;
    void *args[] = {&a};
    // one plane in place at an odd address keeps to its plane bytes; all else
    // of these layouts runs in units, in place those the stream fills whole
    const bool aligned = aligned16(cover) && aligned16(stego);
    // (the aligned kernel's message loads: words or, at k = 3, halves)
    const bool msg_ok = k == 1 || (k == 3 ? a.msg_w2 : a.msg_w4);
    const bool flat = !aligned || !msg_ok;
    if (unit_layout(plane_only, g) && (aligned || !inplace || a.channels == 1) &&
        (!flat || make_flat(cover, stego, C, a.channels, a.plane, false, a.f))) {
        const uint64_t all = plane_only ? (uint64_t)g->width * g->height : C; // carrying bytes
        a.n_carry = inplace ? t_carry : all;
        a.edge_end = inplace ? t_carry * a.channels : C;
        if (!flat) {
            a.f.h = a.f.d = a.f.x0 = 0;
            a.f.ph = a.plane;
            a.f.sel = make_sel(a.channels, a.plane);
            a.f.nunits = a.n_carry >> 4;
        } else if (inplace) {
            const uint64_t whole = t_carry > a.f.x0 ? (t_carry - a.f.x0) >> 4 : 0u;
            if (whole < a.f.nunits)
                a.f.nunits = whole;
            if (a.f.h > a.edge_end)
                a.f.h = (uint32_t)a.edge_end; // (a stream that ends in the head)
        }
        const uint64_t bits0 = (uint64_t)k * a.f.x0; // stream bits before unit 0
        a.full_units = a.t_bits > bits0 ? (a.t_bits - bits0) / (16u * k) : 0u;
        a.part_units = a.t_bits > bits0 ? (a.t_bits - bits0 + 16u * k - 1) / (16u * k) : 0u;
        const void *kern = flat ? (stats ? embed_units_kernel<true, true>(k, a.channels)
                                         : embed_units_kernel<false, true>(k, a.channels))
                                : (stats ? embed_units_kernel<true, false>(k, a.channels)
                                         : embed_units_kernel<false, false>(k, a.channels));
        const int TU = a.channels == 1 ? T : kAsyncThreads; // plane units: the pipeline's CTAs
        const int grid = persistent_grid(kern, TU, 0, kAnyCtas, a.f.nunits ? a.f.nunits : 1,
                                         (uint64_t)TU);
        return launch_counting(kern, dim3(grid), dim3(TU), args, 0, s, stats ? res : nullptr, slot);
    }
    if (plane_only && !inplace) {
        // the non-carrying bytes come from a copy of the cover (a stream
        // embed with nothing to carry), then the plane bytes are rewritten
        cudaError_t e = s1_embed(cover, stego, C, 0, nullptr, 0, false, 0, false, nullptr, 0, sh, s);
        if (e != cudaSuccess)
            return e;
    }
    a.n_carry = plane_only ? t_carry : (inplace ? t_carry : C);
    const void *kern = stats ? (const void *)embedk_bytes<true> : (const void *)embedk_bytes<false>;
    const int grid = persistent_grid(kern, T, 0, kAnyCtas, a.n_carry ? a.n_carry : 1,
                                     (uint64_t)T * 16);
    return launch_counting(kern, dim3(grid), dim3(T), args, 0, s, stats ? res : nullptr, slot);
}

cudaError_t sk_extract(const uint8_t *st, uint64_t C, uint32_t k, bool plane_only,
                       const stego_geom *g, uint8_t *msg, uint64_t cap, uint64_t raw_len,
                       bool header, stego_result *res, const Shape &sh, cudaStream_t s)
{
    KView a;
    std::memset(&a, 0, sizeof(a));
    a.cover = st;
    a.out = msg;
    a.C = C;
    a.cap = cap;
    a.raw_len = raw_len;
    a.k = k;
    a.header = header ? 1u : 0u;
    a.plane_only = plane_only ? 1u : 0u;
    a.channels = plane_only ? g->channels : 1u;
    a.plane = plane_only ? g->plane : 0u;
    a.n_carry = plane_only ? (uint64_t)g->width * g->height : C;
    a.res = res;
    const uint64_t avail_bits = a.n_carry * k;
    uint64_t max_len = raw_len;
    if (header) {
        const uint64_t fit = avail_bits >= 32 ? (avail_bits - 32) / 8 : 0;
        max_len = fit < cap ? fit : cap;
    }
    const int T = sh.threads;
    void *args[] = {&a};
    if (unit_layout(plane_only, g)) {
        const bool flat = !aligned16(st);
        const uint32_t ch = a.channels;
        const uint64_t units = (max_len + 4 + 2 * k - 1) / (2 * k);
        a.f.d = (uint32_t)((uintptr_t)st & 15u);
        a.f.sel = make_sel(ch, a.plane);
        a.f.nunits = a.n_carry >> 4;
        a.u_lo = 0;
        if (flat) {
            // units whose CH + 1 vectors lie inside the stego
            a.u_lo = 1;
            a.f.nunits = C > 16u - a.f.d ? (C - (16u - a.f.d)) / (16u * ch) : 0u;
        }
        const void *kern = flat ? extract_units_kernel<true>(k, ch) : extract_units_kernel<false>(k, ch);
        const int per_thread = ch == 1 ? kExtractAllBytesUnits : 1;
        const int grid = persistent_grid(kern, T, 0, kAnyCtas, units ? units : 1,
                                         (uint64_t)T * per_thread);
        return launch_dependent(kern, dim3(grid), dim3(T), args, 0, s);
    }
    const void *kern = (const void *)extractk_bytes;
    const int grid = persistent_grid(kern, T, 0, kAnyCtas, max_len ? max_len : 1, (uint64_t)T);
    return launch_dependent(kern, dim3(grid), dim3(T), args, 0, s);
}

} // namespace stego

// p2_device.cuh -- device routines of the paper's own layout (Sections VI
// and VII), shared by the single-image kernels (paper2.cu) and the
// persistent batched kernels (batched.cu).
//
// Row r of plane `plane` is A_r[x] = cover[(r*W + x)*channels + plane].  With
// Q = floor(W/4) (Section VI step 5: 4*|B| <= |A|), rows take Q message bytes
// each until fewer than Q remain (Section VII step 4): rows 0..R-2 take Q,
// row R-1 takes L_last = N - (R-1)*Q.  Block i of the paper's launch writes
// bit pair i of B[j] to A_r[L_r*i + j] (Section VI step 7); extraction ORs the
// pairs back (Section VII step 6).
//
// Work units:
//   unit  16 * CH consecutive stego bytes, counted from a 128-byte boundary on
//         (a 16-byte one in an image of less than 16 KiB; CH in {1,3,4}
//         channels): CH whole vectors, which hold the plane bytes of 16
//         consecutive pixels at the same unit bytes everywhere, whatever the
//         row length and the buffers' addresses (see Flat).  One-pass
//         out-of-place embedding (2C + N bytes).
//   run   the message bytes of one row in one 16-byte block of the output:
//         extraction reads the 16 pixels at columns i*L + j of each quarter
//         i as the aligned vectors around them and ORs their pairs.
//   row   thread j of a row handles B[r*Q + j] and its four plane bytes (any
//         channel count; in place; after a copy out of place).
#pragma once

#include "async_copy.cuh"
#include "internal.cuh"
#include "unit_device.cuh"

namespace stego {
namespace p2 {

struct View {
    const uint8_t *src; // cover (embed) or stego (extract)
    uint8_t *dst;       // stego (embed)
    const uint8_t *msg_in;
    uint8_t *msg_out;
    uint64_t N;
    uint32_t W, H, channels, plane;
    uint32_t Q;      // bytes per full row, floor(W/4)
    uint32_t R;      // rows that carry data
    uint32_t L_last; // bytes in row R-1
    uint32_t kmul;   // 4, a multiplier the compiler cannot see (see unit_stats)
};

__host__ __device__ inline View make_view(const uint8_t *src, uint8_t *dst, uint32_t W,
                                          uint32_t H, uint32_t channels, uint32_t plane,
                                          const uint8_t *msg_in, uint8_t *msg_out, uint64_t N)
{
    View v;
    v.src = src;
    v.dst = dst;
    v.msg_in = msg_in;
    v.msg_out = msg_out;
    v.N = N;
    v.W = W;
    v.H = H;
    v.channels = channels;
    v.plane = plane;
    v.Q = W / 4u;
    v.R = v.Q ? (uint32_t)((N + v.Q - 1) / v.Q) : 0u;
    v.L_last = v.R ? (uint32_t)(N - (uint64_t)(v.R - 1) * v.Q) : 0u;
    v.kmul = 4u;
    return v;
}

__device__ __forceinline__ uint32_t row_len(const View &a, uint32_t r)
{
    return r + 1 < a.R ? a.Q : (r + 1 == a.R ? a.L_last : 0u);
}

// Quarter of a carrying column (block i of the paper): 0..3.
__device__ __forceinline__ uint32_t quarter(uint32_t col, uint32_t L)
{
    return (col >= L) + (col >= 2 * L) + (col >= 3 * L);
}

// Quotient of a pixel or run index by a row length: in 32 bits where it fits
// (a 64-bit division is some 100 instructions, a microsecond of a small
// launch).
__device__ __forceinline__ uint32_t row_of(uint64_t x, uint32_t W)
{
    return (x >> 32) == 0 ? (uint32_t)x / W : (uint32_t)(x / W);
}

// The flat units of a cover, at most 2^31 of them (unit indices are counted in
// 32 bits, a grid stride of headroom kept).
__host__ __device__ inline bool plan_units(const uint8_t *cover, const uint8_t *stego, uint64_t C,
                                           uint32_t ch, uint32_t plane, bool lead, Flat &f)
{
    return make_flat(cover, stego, C, ch, plane, lead, f) && f.nunits < (1ull << 31);
}

// Units with carrying pixels: a prefix of the image's units.
__device__ __forceinline__ uint32_t carrying_units(const View &a, const Flat &f)
{
    const uint64_t last = a.R ? (uint64_t)(a.R - 1) * a.W + 4ull * a.L_last : 0ull; // pixels before its end
    const uint64_t n = last > f.x0 ? (last - f.x0 + 15u) / 16u : 0ull;
    return (uint32_t)(n < f.nunits ? n : f.nunits);
}

// (row, column) advanced by dr rows and dc < W columns.
__device__ __forceinline__ void rc_add(uint32_t &r, uint32_t &c, uint32_t dr, uint32_t dc,
                                       uint32_t W)
{
    r += dr;
    if (c >= W - dc) {
        c -= W - dc;
        ++r;
    } else {
        c += dc;
    }
}

// Message bytes off .. off + 15 one by one, 0 outside the message, four loads
// in flight together (a loop, to keep the code of this rare case small).
__device__ __forceinline__ void window_bytes(const uint8_t *__restrict__ msg, uint64_t N,
                                             int64_t off, uint32_t (&m)[4])
{
    m[0] = m[1] = m[2] = m[3] = 0u;
#pragma unroll 1
    for (int q = 0; q < 4; ++q, off += 4) {
        uint32_t b[4];
#pragma unroll
        for (int t = 0; t < 4; ++t)
            b[t] = (uint64_t)(off + t) < N ? (uint32_t)__ldg(msg + (off + t)) : 0u;
        m[0] = m[1];
        m[1] = m[2];
        m[2] = m[3];
        m[3] = __byte_perm(__byte_perm(b[0], b[1], 0x0040u), __byte_perm(b[2], b[3], 0x0040u), 0x5410u);
    }
}

// Message bytes off .. off + 15 as four words: one vector load where they lie
// on a 16-byte boundary, else the five aligned words around them and a funnel
// shift each (rows of W pixels start at any message address when floor(W/4) is
// not a multiple of 4; byte loads took 16 instructions and requests), else,
// where those words are not all inside the message, one by one.
__device__ __forceinline__ void load_window(const uint8_t *__restrict__ msg, uint64_t N,
                                            int64_t off, uint32_t (&m)[4])
{
    const uintptr_t p = (uintptr_t)msg + (uintptr_t)off;
    const uint32_t s = (uint32_t)(p & 3u);
    const uintptr_t w0 = p - s;
    if (off >= 0 && (p & 15u) == 0 && (uint64_t)off + 16u <= N) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p));
        m[0] = v.x;
        m[1] = v.y;
        m[2] = v.z;
        m[3] = v.w;
    } else if (off >= (int64_t)s && (uint64_t)(off - s) + 20u <= N) {
        const uint32_t *w = reinterpret_cast<const uint32_t *>(w0);
        uint32_t v[5];
#pragma unroll
        for (int q = 0; q < 5; ++q)
            v[q] = __ldg(w + q);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            m[q] = __funnelshift_r(v[q], v[q + 1], 8u * s);
    } else {
        window_bytes(msg, N, off, m);
    }
}

// Bytes [t, e) of 16 (byte t%4 of word t/4) as a mask of word q.
__device__ __forceinline__ uint32_t span_mask(uint32_t t, uint32_t e, int q)
{
    const int lo = (int)t - 4 * q, hi = (int)e - 4 * q;
    const uint32_t a = lo <= 0 ? 0xFFFFFFFFu : lo >= 4 ? 0u : 0xFFFFFFFFu << (8 * lo);
    const uint32_t b = hi >= 4 ? 0xFFFFFFFFu : hi <= 0 ? 0u : 0xFFFFFFFFu >> (32 - 8 * hi);
    return a & b;
}

// G[q] takes the low two bits of m[q] >> sh under the byte mask of [t, e).
__device__ __forceinline__ void merge_pairs(uint32_t (&G)[4], const uint32_t (&m)[4], uint32_t sh,
                                            uint32_t t, uint32_t e)
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t k = span_mask(t, e, q);
        G[q] = (G[q] & ~k) | ((m[q] >> sh) & k);
    }
}

// The pairs of 16 pixels that start at (r, col) and do not all lie in one
// quarter of a row; G holds the pixels' plane bytes, whose low two bits the
// pixels that carry nothing keep.  Between full rows of quarters of at least
// 16 pixels there are two spans, the pixels before the end of the quarter and
// those of the next quarter (or, past the at most three columns that carry
// nothing, of the next row), one message window and one masked merge each;
// otherwise quarter by quarter.  At a row length of 5471 one unit in 68 comes
// here, at 1000 one in 12, so that nearly every warp there has one (gray
// 5471x3647: 15.1 us, with the loop alone 16.9).
__device__ __forceinline__ void edge_pairs(const View &a, uint32_t r, uint32_t col,
                                           uint32_t (&G)[4])
{
    uint32_t m[4];
    if (a.Q >= 16u && r + 2 < a.R) {
        const uint32_t i = quarter(col, a.Q);
        const bool carries = col < 4u * a.Q;
        const uint32_t n = carries && (i + 1) * a.Q - col < 16u ? (i + 1) * a.Q - col : 0u;
        const uint64_t row = (uint64_t)r * a.Q;
        if (n) { // the first span
            load_window(a.msg_in, a.N, (int64_t)(row + col - i * a.Q), m);
            merge_pairs(G, m, 2 * i, 0, n);
        }
        // the second: byte 0 of the next quarter, or of the next row
        const bool same = i < 3u;
        const uint32_t t = same ? n : a.W - col;
        load_window(a.msg_in, a.N, (int64_t)(same ? row : row + a.Q) - (int64_t)t, m);
        merge_pairs(G, m, same ? 2 * i + 2 : 0u, t, 16u);
        return;
    }
    uint32_t t = 0;
#pragma unroll 1
    while (t < 16 && r < a.R) {
        const uint32_t L = row_len(a, r), i = quarter(col, L);
        if (col < 4u * L) { // L >= 1 for r < R
            const uint32_t left = (i + 1) * L - col, n = left < 16u - t ? left : 16u - t;
            load_window(a.msg_in, a.N, (int64_t)((uint64_t)r * a.Q + (col - i * L)) - (int64_t)t, m);
            merge_pairs(G, m, 2 * i, t, t + n);
            t += n;
            col += n;
        }
        if (col >= 4u * L) { // the columns past the last quarter carry nothing
            const uint32_t rest = a.W - col;
            t = rest < 16u ? t + rest : 16u;
            col = 0;
            ++r;
        }
    }
}

// What one unit needs besides its cover vectors: how it is embedded (mode 0
// copy only, 1 all 16 pixels in one quarter of a row, 2 otherwise), its first
// pixel (mode 2) and, in mode 1, its shift and 16 message bytes.
struct UnitJob {
    uint32_t mode, r, col, sh;
    uint32_t m[4];
};

__device__ __forceinline__ void plan_unit(const View &a, bool carries, uint32_t r, uint32_t col,
                                          UnitJob &J)
{
    J.mode = 0;
    if (carries) {
        const uint32_t L = row_len(a, r), i = quarter(col, L), e = (i + 1) * L;
        if (col < e && e - col >= 16u) {
            J.mode = 1;
            J.sh = 2 * i;
            load_window(a.msg_in, a.N, (int64_t)((uint64_t)r * a.Q + (col - i * L)), J.m);
        } else {
            J.mode = 2;
            J.r = r;
            J.col = col;
        }
    }
}

// Embeds a planned unit in registers (mode != 0).
template <int CH, bool STATS>
__device__ __forceinline__ void embed_unit(const View &a, const UnitJob &J, const PlaneSel &sel,
                                           uint32_t (&o)[4 * CH], unsigned long long &changed,
                                           unsigned long long &sse)
{
    uint32_t Gn[4], Go[4];
    if (STATS || J.mode == 2)
        get_unit<CH>(o, sel, Go); // old plane bytes
    if (J.mode == 1) {
        // pair of the unit's quarter in the low two bits of each byte
#pragma unroll
        for (int q = 0; q < 4; ++q)
            Gn[q] = J.m[q] >> J.sh;
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            Gn[q] = Go[q];
        edge_pairs(a, J.r, J.col, Gn);
    }
    put_unit<CH>(o, sel, Gn);
    if (STATS) {
        uint32_t d[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            d[q] = (Gn[q] ^ Go[q]) & 0x03030303u;
        unit_stats<2>(Gn, Go, d, a.kmul, changed, sse);
    }
}

// The bytes outside the units, [0, f.h) and [f.h + 16*CH*nunits, C), one per
// thread of the calling CTA; `head` and `tail` choose which.  In place only
// those that change are written.
template <bool STATS>
__device__ __forceinline__ void edge_bytes(const View &a, const Flat &f, bool head, bool tail,
                                           unsigned long long &changed, unsigned long long &sse)
{
    const uint64_t C = (uint64_t)a.W * a.H * a.channels;
    const uint64_t t0 = f.h + 16ull * a.channels * f.nunits;
    const uint32_t nh = head ? f.h : 0u, nt = tail ? (uint32_t)(C - t0) : 0u;
    for (uint32_t e = threadIdx.x; e < nh + nt; e += blockDim.x) {
        const uint64_t k = e < nh ? e : t0 + (e - nh);
        const uint64_t x = a.channels == 1 ? k : a.channels == 4 ? k >> 2 : k / 3u;
        const uint32_t cb = a.src[k];
        uint32_t ob = cb;
        if ((uint32_t)(k - x * a.channels) == a.plane) {
            const uint32_t r = row_of(x, a.W);
            const uint32_t col = (uint32_t)(x - (uint64_t)r * a.W);
            const uint32_t L = r < a.R ? row_len(a, r) : 0u;
            if (col < 4u * L) {
                const uint32_t i = quarter(col, L);
                ob = (cb & 0xFCu) | ((__ldg(a.msg_in + (uint64_t)r * a.Q + (col - i * L)) >> (2 * i)) & 3u);
            }
        }
        if (ob != cb || a.dst != a.src)
            a.dst[k] = (uint8_t)ob;
        if (STATS) {
            const uint32_t d = ob > cb ? ob - cb : cb - ob;
            changed += d != 0;
            sse += d * d;
        }
    }
}

// Shared memory of a units_embed_async CTA of at most 256 threads: two stages
// of a warp's vectors, and the one after them.
constexpr int kStageWarps = 8;
template <int CH>
__host__ __device__ constexpr uint32_t stage_vectors()
{
    return kStageWarps * 2 * (unit_stage_slots<CH>() + 1);
}

// One pass over units k = k_first + i*step < k_end, each thread on its own units:
// every load of a unit (cover, then message) is issued before any arithmetic.  With
// one channel the lanes' single-vector units are consecutive (coalesced); with
// three or four a lane's unit lies 16*CH bytes from its neighbour's, which
// units_embed_async avoids and the batched kernels accept for their register
// budget.  Cover and stego at different addresses mod 16: the vector after the
// unit's own is loaded too (the neighbour's first: an L1 hit) and the bytes joined.
// Out of place every unit is written (units without carrying pixels are copied); in
// place (INPLACE) k_end is cut to the carrying units, each unit read and written
// back by the same thread.  BATCHED: three channels' plane byte at unit byte 0 (see
// plan_units' lead), and a unit's row by a division each: kept from unit to unit by
// additions it costs registers that the batched kernels spill (300 HD frames 645 us,
// so 624; one channel in the single-cover kernel, which does not spill, 31.0
// and 32.1).  SHIFTED = false: the addresses agree mod 16 (f.d = 0).
template <int CH, bool STATS, bool INPLACE = false, bool BATCHED = false, bool SHIFTED = true>
__device__ __forceinline__ void units_embed(const View &a, const Flat &f, uint32_t k_first,
                                            uint32_t k_end, uint32_t step,
                                            unsigned long long &changed, unsigned long long &sse)
{
    const uint32_t carry = carrying_units(a, f);
    if (INPLACE && k_end > carry)
        k_end = carry;
    if (k_first >= k_end)
        return;
    const PlaneSel sel = BATCHED && CH == 3 ? make_sel(3, 0) : f.sel;
    const uint4 *__restrict__ src = reinterpret_cast<const uint4 *>(a.src + f.h - f.d);
    uint4 *dst = reinterpret_cast<uint4 *>(a.dst + f.h);
    // row and column of the unit's first pixel
    const uint64_t x0 = f.x0 + 16ull * k_first;
    uint32_t r = row_of(x0, a.W), col = (uint32_t)(x0 - (uint64_t)r * a.W);
    const uint32_t sr = 16u * step / a.W, sc = 16u * step - sr * a.W; // 16 * step < 2^32
    for (uint32_t k = k_first; k < k_end; k += step) {
        uint32_t c[4 * CH + 4], o[4 * CH];
#pragma unroll
        for (int q = 0; q < CH; ++q)
            set_vec(c, q, __ldcs(src + (uint64_t)k * CH + q));
        if (SHIFTED && !INPLACE && f.d)
            set_vec(c, CH, __ldcs(src + (uint64_t)k * CH + CH));
        if constexpr (BATCHED) {
            const uint64_t x = f.x0 + 16ull * k;
            r = row_of(x, a.W);
            col = (uint32_t)(x - (uint64_t)r * a.W);
        }
        UnitJob J;
        plan_unit(a, k < carry, r, col, J);
        if (SHIFTED && !INPLACE && f.d) {
            join_unit<CH>(c, f.d, o);
        } else {
#pragma unroll
            for (int q = 0; q < 4 * CH; ++q)
                o[q] = c[q];
        }
        if (J.mode)
            embed_unit<CH, STATS>(a, J, sel, o, changed, sse);
#pragma unroll
        for (int q = 0; q < CH; ++q)
            __stcs(dst + (uint64_t)k * CH + q, get_vec(o, q));
        if constexpr (!BATCHED)
            rc_add(r, col, sr, sc, a.W);
    }
}

// units_embed for CH > 1 with a two-stage copy pipeline per warp: while the
// warp embeds its 32 units from shared memory, the cover vectors of its next
// 32 are already on their way there (cp.async, memory order, coalesced) and
// the next units' message bytes on their way to registers.  SHIFTED: cover and
// stego at different addresses mod 16 (f.d != 0); the stage then holds the
// 32*CH + 1 aligned cover vectors around the warp's bytes, of which each lane
// reads CH + 1.  Same results as units_embed; `stage` is the CTA's
// stage_vectors<CH>() vectors of shared memory.
template <int CH, bool STATS, bool SHIFTED, bool INPLACE = false>
__device__ __forceinline__ void units_embed_async(const View &a, const Flat &f, uint32_t k_first,
                                                  uint32_t k_end, uint32_t step,
                                                  unsigned long long &changed,
                                                  unsigned long long &sse, uint4 *stage)
{
    static_assert(CH > 1, "one-channel units are single vectors, loaded coalesced as they are");
    const uint32_t carry = carrying_units(a, f);
    if (INPLACE && k_end > carry)
        k_end = carry;
    const uint4 *__restrict__ src = reinterpret_cast<const uint4 *>(a.src + f.h - (SHIFTED ? f.d : 0u));
    uint4 *dst = reinterpret_cast<uint4 *>(a.dst + f.h);
    const uint32_t lane = threadIdx.x & 31u;
    constexpr uint32_t SV = unit_stage_slots<CH>() + (SHIFTED ? 1u : 0u);
    uint4 *const sw = stage + (threadIdx.x >> 5) * 2 * SV;
    const uint64_t vend = (uint64_t)k_end * CH;
    uint32_t k0 = k_first; // the lane's first unit; k0 - lane is the same for the warp
    if (k0 - lane >= k_end)
        return;
    const uint64_t x = f.x0 + 16ull * k_first;
    uint32_t r0 = row_of(x, a.W), c0 = (uint32_t)(x - (uint64_t)r0 * a.W);
    const uint32_t sr = 16u * step / a.W, sc = 16u * step - sr * a.W; // 16 * step < 2^32

    // the warp's vectors from lane 0's unit kb on -> stage s
    auto issue = [&](uint32_t kb, uint32_t s) {
        const uint64_t v0 = (uint64_t)kb * CH;
#pragma unroll
        for (int j = 0; j < CH; ++j)
            if (v0 + 32u * j + lane < vend + (SHIFTED ? 1u : 0u))
                cp_async16(sw + s * SV + unit_stage_slot<CH>(32u * j + lane), src + v0 + 32u * j + lane);
        if (SHIFTED && lane == 0 && v0 + 32u * CH <= vend)
            cp_async16(sw + s * SV + unit_stage_slot<CH>(32u * CH), src + v0 + 32u * CH);
        cp_async_commit();
    };

    UnitJob J;
    issue(k0 - lane, 0);
    plan_unit(a, k0 < k_end && k0 < carry, r0, c0, J);
    uint32_t s = 0;
    for (;;) {
        const uint32_t kn = k0 + step;
        const bool next = kn - lane < k_end; // kn < 2^32: units and steps stay below 2^31
        UnitJob Jn;
        if (next) {
            rc_add(r0, c0, sr, sc, a.W);
            issue(kn - lane, s ^ 1u);
            plan_unit(a, kn < k_end && kn < carry, r0, c0, Jn);
            cp_async_wait<1>(); // this iteration's copies landed (the next may be pending)
        } else {
            cp_async_wait<0>();
        }
        __syncwarp(); // every lane's copies visible to the warp
        uint4 *const st = sw + s * SV;
        if constexpr (SHIFTED) {
            uint32_t o[4 * CH];
            if (k0 < k_end) {
                uint32_t v[4 * CH + 4];
#pragma unroll
                for (int q = 0; q <= CH; ++q)
                    set_vec(v, q, st[unit_stage_slot<CH>(CH * lane + q)]);
                join_unit<CH>(v, f.d, o);
                if (J.mode)
                    embed_unit<CH, STATS>(a, J, f.sel, o, changed, sse);
            }
            __syncwarp(); // the neighbour has read this lane's first vector
            if (k0 < k_end) {
#pragma unroll
                for (int q = 0; q < CH; ++q)
                    st[unit_stage_slot<CH>(CH * lane + q)] = get_vec(o, q);
            }
        } else if (k0 < k_end && J.mode) {
            uint32_t o[4 * CH];
#pragma unroll
            for (int q = 0; q < CH; ++q)
                set_vec(o, q, st[unit_stage_slot<CH>(CH * lane + q)]);
            embed_unit<CH, STATS>(a, J, f.sel, o, changed, sse);
#pragma unroll
            for (int q = 0; q < CH; ++q)
                st[unit_stage_slot<CH>(CH * lane + q)] = get_vec(o, q);
        }
        __syncwarp(); // the rewritten units visible to the storing lanes
        const uint64_t v0 = (uint64_t)(k0 - lane) * CH;
#pragma unroll
        for (int j = 0; j < CH; ++j)
            if (v0 + 32u * j + lane < vend)
                __stcs(dst + v0 + 32u * j + lane, st[unit_stage_slot<CH>(32u * j + lane)]);
        if (!next)
            break;
        // stage s is refilled two iterations on, after every lane passed the
        // barriers above and read its own memory-order slots
        J = Jn;
        k0 = kn;
        s ^= 1u;
    }
}

// Scatter of carrying rows r = r_first + i*r_step < min(r_end, R): the
// calling CTA's threads split each row's L message bytes, four per thread in
// flight; each reads B[r*Q + j] once and rewrites its four plane bytes (from
// src into dst; src may equal dst).
template <bool STATS>
__device__ __forceinline__ void rows_embed(const View &a, uint32_t r_first, uint32_t r_end,
                                           uint32_t r_step, unsigned long long &changed,
                                           unsigned long long &sse)
{
    const uint32_t rend = r_end < a.R ? r_end : a.R;
    for (uint32_t r = r_first; r < rend; r += r_step) {
        const uint32_t L = row_len(a, r);
        const uint8_t *mrow = a.msg_in + (uint64_t)r * a.Q;
        const uint64_t prow = (uint64_t)r * a.W;
        const uint64_t qstride = (uint64_t)L * a.channels; // pair i at base(j) + i*qstride
        constexpr int U = 4;
        for (uint32_t j0 = threadIdx.x; j0 < L; j0 += blockDim.x * U) {
            uint32_t B[U], c[U][4];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t j = j0 + u * blockDim.x;
                if (j >= L)
                    continue;
                B[u] = __ldg(mrow + j);
                const uint8_t *p = a.src + (prow + j) * a.channels + a.plane;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    c[u][i] = p[i * qstride]; // plain load: src may equal dst (in place)
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t j = j0 + u * blockDim.x;
                if (j >= L)
                    continue;
                uint8_t *p = a.dst + (prow + j) * a.channels + a.plane;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t v = (c[u][i] & 0xFCu) | ((B[u] >> (2 * i)) & 3u);
                    p[i * qstride] = (uint8_t)v;
                    if (STATS) {
                        const uint32_t d = v > c[u][i] ? v - c[u][i] : c[u][i] - v;
                        changed += d != 0;
                        sse += d * d;
                    }
                }
            }
        }
    }
}

// Copy of whole rows [r0, r1) from src to dst by the calling CTA (16-byte
// vectors where src and dst agree modulo 16, bytes otherwise).
__device__ __forceinline__ void rows_copy(const View &a, uint32_t r0, uint32_t r1)
{
    const uint64_t rb = (uint64_t)a.W * a.channels;
    const uint64_t b0 = r0 * rb, b1 = r1 * rb;
    const uint8_t *s = a.src;
    uint8_t *d = a.dst;
    const uint32_t ms = (uint32_t)((uintptr_t)(s + b0) & 15u);
    if (ms == ((uintptr_t)(d + b0) & 15u)) {
        const uint64_t head = ms ? 16u - ms : 0u;
        const uint64_t vb = b0 + head < b1 ? b0 + head : b1;          // first vector byte
        const uint64_t ve = vb + ((b1 - vb) & ~15ull);                // end of whole vectors
        for (uint64_t k = b0 + threadIdx.x; k < vb; k += blockDim.x)
            d[k] = s[k];
        const uint4 *sv = reinterpret_cast<const uint4 *>(s + vb);
        uint4 *dv = reinterpret_cast<uint4 *>(d + vb);
        const uint64_t nv = (ve - vb) >> 4;
        for (uint64_t k = threadIdx.x; k < nv; k += blockDim.x)
            __stcs(dv + k, __ldcs(sv + k));
        for (uint64_t k = ve + threadIdx.x; k < b1; k += blockDim.x)
            d[k] = s[k];
    } else {
        for (uint64_t k = b0 + threadIdx.x; k < b1; k += blockDim.x)
            d[k] = s[k];
    }
}

// Runs of an extraction: row r's message bytes lie in at most run_row()
// 16-byte blocks of the output, counted from the block that holds its first
// byte; run k is block k mod run_row() of row k / run_row().  A run takes the
// bytes of its block that are its row's: all 16 but in the row's first and
// last block, which it shares with the neighbouring rows' runs.
// Where rows and quarters of the image and rows of the output are whole
// 16-byte vectors (runs_aligned: W a multiple of 64, both buffers 16-byte
// aligned), every run of a full row reads aligned vectors and writes one.
__host__ __device__ inline bool runs_aligned(const View &v)
{
    return v.W % 64u == 0 && (((uintptr_t)v.src | (uintptr_t)v.msg_out) & 15u) == 0;
}

__host__ __device__ inline uint32_t run_row(const View &v)
{
    return runs_aligned(v) ? v.Q / 16u : (uint32_t)(((uint64_t)v.Q + 30u) / 16u);
}

__host__ __device__ inline uint64_t run_count(const View &v)
{
    return v.Q ? (uint64_t)v.R * run_row(v) : 0u;
}

// Quarter i's plane bytes P into M: pair t in bits 2i of byte t.
__device__ __forceinline__ void take_pairs(uint32_t (&M)[4], const uint32_t (&P)[4], int i)
{
#pragma unroll
    for (int q = 0; q < 4; ++q)
        M[q] |= (P[q] & 0x03030303u) << (2 * i);
}

// The pairs of the 16 pixels whose first plane byte is byte `off` of the image,
// for G quarters from i0 on, `stride` bytes apart.  Each is read as the CH (on a
// 16-byte boundary) or CH + 1 aligned vectors around its bytes where those lie
// inside the image, else byte by byte, pixels [t, e) alone.
template <int CH, int G>
__device__ __forceinline__ void run_quarters(const View &a, uint64_t C, int64_t off,
                                             uint64_t stride, int i0, uint32_t t, uint32_t e,
                                             uint32_t (&M)[4])
{
    const uintptr_t lo = (uintptr_t)a.src, hi = lo + C;
    uint32_t v[G][4 * CH + 4];
    bool whole[G];
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const uintptr_t p = lo + (uintptr_t)(off + (int64_t)((i0 + i) * stride));
        const uint32_t d = (uint32_t)(p & 15u);
        const uint4 *A = reinterpret_cast<const uint4 *>(p - d);
        whole[i] = p - d >= lo && p - d + 16u * (CH + (d ? 1u : 0u)) <= hi;
        if (whole[i]) {
#pragma unroll
            for (int q = 0; q < CH; ++q)
                set_vec(v[i], q, __ldg(A + q));
            if (d)
                set_vec(v[i], CH, __ldg(A + CH));
        }
    }
#pragma unroll
    for (int i = 0; i < G; ++i) {
        uint32_t P[4];
        const int64_t at = off + (int64_t)((i0 + i) * stride);
        if (whole[i]) {
            const uint32_t d = (uint32_t)((lo + (uintptr_t)at) & 15u);
            uint32_t c[4 * CH];
            if (d) {
                join_unit<CH>(v[i], d, c);
            } else {
#pragma unroll
                for (int q = 0; q < 4 * CH; ++q)
                    c[q] = v[i][q];
            }
            get_unit<CH>(c, make_sel(CH, 0), P);
        } else {
            const uint8_t *p = a.src + at;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t b[4];
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    b[x] = 4u * q + x >= t && 4u * q + x < e ? (uint32_t)__ldg(p + (4 * q + x) * CH) : 0u;
                P[q] = __byte_perm(__byte_perm(b[0], b[1], 0x0040u),
                                   __byte_perm(b[2], b[3], 0x0040u), 0x5410u);
            }
        }
        take_pairs(M, P, i0 + i);
    }
}

// Pairs of the plane bytes of a unit's words (pair t in byte t%4 of P[t/4]), one
// shift and one masked merge per pixel: with the byte position at compile time
// faster here than gathering by byte_perm.
template <int CH, int PLANE>
__device__ __forceinline__ void get_pairs(const uint32_t (&w)[4 * CH], uint32_t (&P)[4])
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        P[q] = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int at = (4 * q + j) * CH + PLANE;
            P[q] |= ((w[at >> 2] >> (8 * (at & 3))) & 3u) << (8 * j);
        }
    }
}

// Runs k = k_first + i*step < k_end of an aligned layout's full rows, GA
// quarters' vectors at a time.  BATCHED: a run's row and block by a 32-bit division,
// else kept by additions (8192x8192x3 33.1 us, 33.4 by divisions; in the batched
// kernel the additions cost registers that it spills: 1024 paper covers 380 us, by
// divisions here and in other_runs 372), the step in rows and blocks found when there
// is a next run: a launch of one run per thread is a chain of latencies, in which
// that division and one for the first run after these were 0.4 of 2.0 us (gray
// 1920x1080).  Returns the first k that it did not take.
template <int CH, int PLANE, int GA, bool BATCHED>
__device__ __forceinline__ uint64_t full_runs(const View &a, uint64_t k_first, uint64_t k_end,
                                          uint32_t step)
{
    const uint32_t rpr = a.Q / 16u, W16 = a.W / 16u;
    const uint32_t stride = rpr * CH; // vectors from quarter to quarter
    uint32_t r = row_of(k_first, rpr), b = (uint32_t)(k_first - (uint64_t)r * rpr);
    uint32_t dr = 0, db = 0; // (step > 0: not both, once known)
    const uint4 *__restrict__ src = reinterpret_cast<const uint4 *>(a.src);
    uint4 *out = reinterpret_cast<uint4 *>(a.msg_out);
    uint64_t k = k_first;
    while (k < k_end) {
        if constexpr (BATCHED) {
            r = row_of(k, rpr);
            b = (uint32_t)(k - (uint64_t)r * rpr);
        }
        const uint4 *A = src + ((uint64_t)r * W16 + b) * CH;
        uint32_t M[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int i = 0; i < 4; i += GA) {
            uint32_t v[GA][4 * CH];
#pragma unroll
            for (int x = 0; x < GA; ++x)
#pragma unroll
                for (int q = 0; q < CH; ++q)
                    set_vec(v[x], q, __ldcs(A + (uint64_t)(i + x) * stride + q));
#pragma unroll
            for (int x = 0; x < GA; ++x) {
                uint32_t P[4];
                if constexpr (CH == 1) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        P[q] = v[x][q] & 0x03030303u;
                } else {
                    get_pairs<CH, PLANE>(v[x], P);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    M[q] |= P[q] << (2 * (i + x));
            }
        }
        out[k] = make_uint4(M[0], M[1], M[2], M[3]);
        k += step;
        if constexpr (!BATCHED) {
            if (k >= k_end)
                break;
            if ((dr | db) == 0) {
                dr = step / rpr;
                db = step - dr * rpr;
            }
            rc_add(r, b, dr, db, rpr);
        }
    }
    return k;
}

// Runs k = k_first + i*step < k_end of any layout, G quarters' vectors at a time
// (BATCHED: see full_runs).
template <int CH, int G, bool BATCHED>
__device__ __forceinline__ void other_runs(const View &a, uint64_t k_first, uint64_t k_end,
                                           uint32_t step)
{
    const uint32_t rpr = run_row(a);
    uint32_t r = row_of(k_first, rpr), b = (uint32_t)(k_first - (uint64_t)r * rpr);
    uint32_t dr = 0, db = 0;
    const uint64_t C = (uint64_t)a.W * a.H * CH;
    for (uint64_t k = k_first; k < k_end; k += step) {
        if constexpr (BATCHED) {
            r = row_of(k, rpr);
            b = (uint32_t)(k - (uint64_t)r * rpr);
        }
        const uint32_t L = row_len(a, r);
        uint8_t *mrow = a.msg_out + (uint64_t)r * a.Q;
        const int64_t j0 = 16ll * b - (int64_t)((uintptr_t)mrow & 15u); // row byte of the block's first
        if (j0 < (int64_t)L) {
            const uint32_t t = j0 < 0 ? (uint32_t)-j0 : 0u;
            const uint32_t e = (int64_t)L - j0 < 16 ? (uint32_t)(L - j0) : 16u;
            const int64_t off = ((int64_t)((uint64_t)r * a.W) + j0) * CH + a.plane;
            uint32_t M[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int i = 0; i < 4; i += G)
                run_quarters<CH, G>(a, C, off, (uint64_t)L * CH, i, t, e, M);
            uint8_t *mp = mrow + j0;
            if (e - t == 16u) {
                *reinterpret_cast<uint4 *>(mp) = make_uint4(M[0], M[1], M[2], M[3]);
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (t <= 4u * q && e >= 4u * q + 4u) {
                        reinterpret_cast<uint32_t *>(mp)[q] = M[q];
                    } else {
#pragma unroll
                        for (uint32_t x = 4u * q; x < 4u * q + 4u; ++x)
                            if (x >= t && x < e)
                                mp[x] = (uint8_t)(M[q] >> (8 * (x & 3u)));
                    }
                }
            }
        }
        if constexpr (!BATCHED) {
            if (k + step >= k_end)
                break;
            if ((dr | db) == 0) {
                dr = step / rpr;
                db = step - dr * rpr;
            }
            rc_add(r, b, dr, db, rpr);
        }
    }
}

// Runs of an aligned layout's full rows.
__host__ __device__ inline uint64_t aligned_full_runs(const View &a)
{
    return (uint64_t)(a.L_last == a.Q ? a.R : a.R - 1) * (a.Q / 16u);
}

// full_runs of the cover's plane.
template <int CH, int GA, bool BATCHED>
__device__ __forceinline__ uint64_t aligned_runs(const View &a, uint64_t k_first, uint64_t k_end,
                                             uint32_t step)
{
    switch (CH == 1 ? 0u : a.plane) {
    case 0: return full_runs<CH, 0, GA, BATCHED>(a, k_first, k_end, step);
    case 1: return full_runs<CH, CH == 1 ? 0 : 1, GA, BATCHED>(a, k_first, k_end, step);
    case 2: return full_runs<CH, CH == 1 ? 0 : 2, GA, BATCHED>(a, k_first, k_end, step);
    default: return full_runs<CH, CH == 4 ? 3 : 0, GA, BATCHED>(a, k_first, k_end, step);
    }
}

// Extraction over runs k = k_first + i*step < k_end: those of an aligned layout's
// full rows GA quarters' vectors at a time, then all others G.
template <int CH, int GA, int G>
__device__ __forceinline__ void runs_extract(const View &a, uint64_t k_first, uint64_t k_end,
                                             uint32_t step)
{
    if (k_first >= k_end)
        return;
    if (runs_aligned(a)) {
        const uint64_t full = aligned_full_runs(a);
        k_first = aligned_runs<CH, GA, false>(a, k_first, k_end < full ? k_end : full, step);
        if (k_first >= k_end)
            return;
    }
    other_runs<CH, G, false>(a, k_first, k_end, step);
}

// Extraction of carrying rows r = r_first + i*r_step < min(r_end, R), any
// channel count: the calling CTA's threads split each row's L bytes.
__device__ __forceinline__ void rows_extract(const View &a, uint32_t r_first, uint32_t r_end,
                                             uint32_t r_step)
{
    const uint32_t rend = r_end < a.R ? r_end : a.R;
    for (uint32_t r = r_first; r < rend; r += r_step) {
        const uint32_t L = row_len(a, r);
        uint8_t *mrow = a.msg_out + (uint64_t)r * a.Q;
        const uint64_t prow = (uint64_t)r * a.W;
        constexpr int U = 4;
        for (uint32_t j0 = threadIdx.x; j0 < L; j0 += blockDim.x * U) {
            uint32_t c[U][4];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t j = j0 + u * blockDim.x;
                if (j >= L)
                    continue;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    c[u][i] = __ldg(a.src + (prow + (uint64_t)L * i + j) * a.channels + a.plane);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t j = j0 + u * blockDim.x;
                if (j >= L)
                    continue;
                uint32_t B = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    B |= (c[u][i] & 3u) << (2 * i);
                mrow[j] = (uint8_t)B;
            }
        }
    }
}

// The layouts the unit and run routines handle.
__host__ __device__ inline bool unit_channels(uint32_t ch) { return ch == 1 || ch == 3 || ch == 4; }

} // namespace p2
} // namespace stego

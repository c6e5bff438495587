// stats.cu -- changed-byte count and squared error of two byte arrays, the
// integer quantities behind the PSNR that Section VIII reports:
//   changed = #{k : a[k] != b[k]},  sse = sum (a[k] - b[k])^2,
//   MSE = sse / n,  PSNR = 10 log10(255^2 / MSE).
// Both are exact (64-bit integer accumulation); the host turns them into
// PSNR.  A standalone pass reads 2n bytes; the embed kernels fuse statistics of
// their own into their store loop at no extra traffic.
#include "s1_device.cuh"

namespace stego {
namespace {

// Changed bytes and squared error of 16 byte pairs, added in 32 bits (at most
// 16 and 16 * 255^2).  A byte differs when its top bit does or its low seven
// bits of the difference plus 127 carry into it.
__device__ __forceinline__ void vec_stats(const uint4 &x, const uint4 &y, uint32_t &changed,
                                          uint32_t &sse)
{
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
    uint32_t f = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t d = xs[i] ^ ys[i];
        f |= ((((d & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | d) & 0x80808080u) >> i;
        const uint32_t a = __vabsdiffu4(xs[i], ys[i]);
        sse = __dp4a(a, a, sse);
    }
    changed += __popc(f);
}

// Bytes k = threadIdx.x + i*blockDim.x of [b0, b1) by the calling CTA.
__device__ __forceinline__ void byte_stats(const uint8_t *a, const uint8_t *b, uint64_t b0,
                                           uint64_t b1, unsigned long long &changed,
                                           unsigned long long &sse)
{
    for (uint64_t k = b0 + threadIdx.x; k < b1; k += blockDim.x) {
        const uint32_t p = a[k], q = b[k];
        const uint32_t d = p > q ? p - q : q - p;
        changed += d != 0;
        sse += d * d;
    }
}

// Both totals into out[0..1]: through the stream's slot, or into zeroed words.
__device__ __forceinline__ void put_totals(unsigned long long changed, unsigned long long sse,
                                           unsigned long long *out, StatSlot *slot)
{
    // block_stats writes the two totals alone, a result's first two fields
    block_stats(changed, sse, reinterpret_cast<stego_result *>(out), slot);
}

// Both arrays 16-byte aligned: HBM-bound, 8192x8192x3 59.6 us (61.2 with the
// totals of every word added in 64 bits and the result zeroed by a memset
// first; 512x512x3 5.8 -> 4.2 us).
template <int V>
__global__ void __launch_bounds__(512) changed_vec(const uint4 *__restrict__ a,
                                                    const uint4 *__restrict__ b, uint64_t nvec,
                                                    const uint8_t *a8, const uint8_t *b8,
                                                    uint64_t n, unsigned long long *out,
                                                    StatSlot *slot)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    unsigned long long changed = 0, sse = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x * V;
    for (uint64_t v0 = (uint64_t)blockIdx.x * blockDim.x * V + threadIdx.x; v0 < nvec;
         v0 += stride) {
        uint4 x[V], y[V];
#pragma unroll
        for (int u = 0; u < V; ++u) {
            const uint64_t v = v0 + (uint64_t)u * blockDim.x;
            if (v < nvec) {
                x[u] = __ldcs(a + v);
                y[u] = __ldcs(b + v);
            }
        }
        uint32_t c = 0, e = 0;
#pragma unroll
        for (int u = 0; u < V; ++u) {
            const uint64_t v = v0 + (uint64_t)u * blockDim.x;
            if (v < nvec)
                vec_stats(x[u], y[u], c, e);
        }
        changed += c;
        sse += e;
    }
    if (blockIdx.x == 0)
        byte_stats(a8, b8, nvec << 4, n, changed, sse);
    put_totals(changed, sse, out, slot);
}

// Arrays that are not both 16-byte aligned: a in aligned vectors from byte h
// on (a 128-byte boundary of it), b as the aligned vectors around the same
// bytes, which start d bytes into them (d = 4Q + the selector's b; Q = 4: at
// the same address mod 16, d = 0, its own vectors).  Warps take rounds of 32*V
// consecutive vectors, a lane loading one vector of b per vector of a and
// taking the next from its neighbour (s1::next_vec).  HBM-bound: 5471x3647x3
// against a copy at another address 21.0 us, as fast as aligned arrays; with
// single bytes loaded by every thread 102 us (3839x2159x3: 48.5 -> 11.7 us).
template <int Q, int V>
__global__ void __launch_bounds__(512) changed_shift(const uint8_t *a8, const uint8_t *b8,
                                                      uint64_t n, uint32_t h, uint32_t d,
                                                      uint64_t nvec, unsigned long long *out,
                                                      StatSlot *slot)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    unsigned long long changed = 0, sse = 0;
    const uint4 *__restrict__ A = reinterpret_cast<const uint4 *>(a8 + h);
    const uint4 *__restrict__ B = reinterpret_cast<const uint4 *>(b8 + h - d);
    const uint32_t sel = 0x3210u + 0x1111u * (d & 3u);
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t r = warp * 32u * V; r < nvec; r += nwarps * 32u * V) {
        uint4 x[V], y[V], end = make_uint4(0u, 0u, 0u, 0u);
        const bool whole = r + 32u * V <= nvec;
        uint32_t c = 0, e = 0;
        if (whole) {
#pragma unroll
            for (int u = 0; u < V; ++u) {
                x[u] = __ldcs(A + r + 32u * u + lane);
                y[u] = __ldcs(B + r + 32u * u + lane);
            }
            if (Q < 4 && lane == 0)
                end = __ldcs(B + r + 32u * V);
#pragma unroll
            for (int u = 0; u < V; ++u) {
                if constexpr (Q < 4)
                    vec_stats(x[u], s1::funnel16<Q>(y[u], s1::next_vec<V>(y, end, u, lane), sel), c, e);
                else
                    vec_stats(x[u], y[u], c, e);
            }
        } else {
#pragma unroll 1
            for (uint64_t j = r + lane; j < nvec; j += 32u) {
                if constexpr (Q < 4)
                    vec_stats(__ldcs(A + j), s1::funnel16<Q>(__ldcs(B + j), __ldcs(B + j + 1), sel), c, e);
                else
                    vec_stats(__ldcs(A + j), __ldcs(B + j), c, e);
            }
        }
        changed += c;
        sse += e;
    }
    if (blockIdx.x == gridDim.x - 1) { // the CTA with the fewest vectors: the bytes around them
        byte_stats(a8, b8, 0, h, changed, sse);
        byte_stats(a8, b8, h + (nvec << 4), n, changed, sse);
    }
    put_totals(changed, sse, out, slot);
}

// Arrays of less than a few vectors.
__global__ void __launch_bounds__(512) changed_bytes_kernel(const uint8_t *a, const uint8_t *b,
                                                             uint64_t n, unsigned long long *out,
                                                             StatSlot *slot)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    unsigned long long changed = 0, sse = 0;
    byte_stats(a, b, 0, n, changed, sse);
    put_totals(changed, sse, out, slot);
}

constexpr int kShiftV = 4; // vectors in flight per thread of changed_shift
constexpr uint64_t kBytesMost = 1024; // arrays the byte kernel's one CTA takes

} // namespace

cudaError_t changed_bytes(const uint8_t *a, const uint8_t *b, uint64_t n,
                          unsigned long long *out2, const Shape &sh, cudaStream_t s,
                          StatSlot *slot)
{
    const int T = sh.threads;
    if ((((uintptr_t)a | (uintptr_t)b) & 15u) == 0) {
        const uint64_t nvec = n >> 4;
        const void *k;
        switch (sh.vec) {
        case 1: k = (const void *)changed_vec<1>; break;
        case 2: k = (const void *)changed_vec<2>; break;
        case 8: k = (const void *)changed_vec<8>; break;
        default: k = (const void *)changed_vec<4>; break;
        }
        const int vec = (sh.vec == 1 || sh.vec == 2 || sh.vec == 8) ? sh.vec : 4;
        const int grid = persistent_grid(k, T, 0, sh.ctas_per_sm, nvec > 0 ? nvec : 1,
                                         (uint64_t)T * vec);
        const uint4 *av = reinterpret_cast<const uint4 *>(a);
        const uint4 *bv = reinterpret_cast<const uint4 *>(b);
        void *args[] = {&av, &bv, (void *)&nvec, &a, &b, &n, &out2, &slot};
        return launch_counting(k, dim3(grid), dim3(T), args, 0, s, out2, slot);
    }
    if (n <= kBytesMost) {
        void *args[] = {&a, &b, &n, &out2, &slot};
        return launch_counting((const void *)changed_bytes_kernel, dim3(1), dim3(T), args, 0, s, out2, slot);
    }
    // from byte h on a's vectors and the vectors around b's bytes lie inside
    // the arrays (n > kBytesMost leaves room for h and a vector more)
    uint32_t h = (uint32_t)(-(uintptr_t)a & 127u);
    const uint32_t d = (uint32_t)(((uintptr_t)b + h) & 15u);
    if (h < d)
        h += 128u;
    const uint64_t nvec = (n - h - (d ? 16u - d : 0u)) >> 4;
    const void *k;
    switch (d ? d >> 2 : 4u) {
    case 0: k = (const void *)changed_shift<0, kShiftV>; break;
    case 1: k = (const void *)changed_shift<1, kShiftV>; break;
    case 2: k = (const void *)changed_shift<2, kShiftV>; break;
    case 3: k = (const void *)changed_shift<3, kShiftV>; break;
    default: k = (const void *)changed_shift<4, kShiftV>; break;
    }
    const int grid = persistent_grid(k, T, 0, sh.ctas_per_sm, nvec, (uint64_t)T * kShiftV);
    void *args[] = {&a, &b, &n, &h, (void *)&d, (void *)&nvec, &out2, &slot};
    return launch_counting(k, dim3(grid), dim3(T), args, 0, s, out2, slot);
}

} // namespace stego

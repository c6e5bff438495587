// paper2.cu -- single-image kernels of the paper's own layout (Sections VI
// and VII: one plane, two bits per cover byte, the message divided greedily
// among rows, pair i of B[j] at A[L*i + j]).  The per-unit, per-run and
// per-row routines live in p2_device.cuh and are shared with the batched
// kernels.
//   p2_embed_units<CH,STATS,INPLACE,SHIFTED>  persistent grid over flat
//       units (16*CH stego bytes, see Flat); 256-thread CTAs,
//       each warp's units copied to shared memory one iteration ahead
//       (cp.async).  Out of place one pass (2C + N bytes) for any row length
//       and any addresses; in place the units with carrying pixels, read and
//       written back whole.
//   p2_embed_rows  the scatter after a copy (and in place) for layouts the
//       unit kernel does not take; CTAs stride over carrying rows.
//   p2_extract_units<CH>  runs of 16 message bytes (CH in {1,3,4}).
//   p2_extract_rows  any channel count.
#include <cstring>

#include "p2_device.cuh"

namespace stego {
namespace {

// The installed launch shapes are tuned for the one-bit kernels; these
// kernels (other register counts) take as many resident CTAs as occupancy
// allows instead of a tuned CTA count.
constexpr int kAnyCtas = 0;

using p2::View;

struct P2Args {
    View v;
    Flat f;
    stego_result *res;
    StatSlot *slot;
};

__device__ __forceinline__ void write_res(const P2Args &a, bool stats)
{
    if (a.res && blockIdx.x == 0 && threadIdx.x == 0) {
        a.res->msg_bytes = a.v.N;
        a.res->status = STEGO_OK;
        a.res->reserved = 0;
        if (!stats) {
            a.res->changed = 0;
            a.res->sse = 0;
        }
    }
}

constexpr int kUnitThreads = 256; // at most 256: the staging area holds 8 warps

// Out of place every unit of the image; in place the units with carrying
// pixels.  Three or four channels run the two-stage copy pipeline
// (units_embed_async), three CTAs per SM with three channels; one channel
// loads its single-vector units directly, one per thread and five CTAs per SM
// (two per thread in two CTAs: 8192x8192 37.1 us, this 30.8).  HBM-bound where
// the rows are long (8192x8192x3 65.8 us, 0.96 of the measured copy rate);
// the units that cross a quarter or a row (edge_pairs) cost a warp a second
// pass over its units, so that short rows are bound by instructions.  Rows
// that are not whole vectors took a copy and one thread per plane byte before:
// 5471x3647x3 47.5 -> 24.1 us, one channel 28.3 -> 16.4, four 65.9 -> 31.1,
// cover 3 bytes past a boundary 53.6 -> 25.4.  Whole-vector rows of one channel lose
// where there are no statistics (8192x8192 23.6 -> 26.4 us; with them 28.9 as
// before): neither more units in flight (26.4-28), other CTAs (26.1-28) nor a
// kernel of their own for aligned addresses wins it back.
template <int CH, bool STATS, bool INPLACE, bool SHIFTED>
__global__ void __launch_bounds__(kUnitThreads, CH == 4 ? 2 : CH == 1 ? 5 : 3) p2_embed_units(P2Args a)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    unsigned long long changed = 0, sse = 0;
    write_res(a, STATS);
    if (blockIdx.x == gridDim.x - 1) // the CTA with the fewest units
        p2::edge_bytes<STATS>(a.v, a.f, true, true, changed, sse);
    if constexpr (CH > 1) {
        __shared__ uint4 stage[p2::stage_vectors<CH>()];
        p2::units_embed_async<CH, STATS, SHIFTED, INPLACE>(
            a.v, a.f, blockIdx.x * blockDim.x + threadIdx.x, (uint32_t)a.f.nunits, gridDim.x * blockDim.x,
            changed, sse, stage);
    } else {
        p2::units_embed<CH, STATS, INPLACE, false, SHIFTED>(a.v, a.f, blockIdx.x * blockDim.x + threadIdx.x,
                                            (uint32_t)a.f.nunits, gridDim.x * blockDim.x, changed, sse);
    }
    if (STATS)
        block_stats(changed, sse, a.res, a.slot);
}

template <bool STATS>
__global__ void __launch_bounds__(512, 2) p2_embed_rows(P2Args a)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    unsigned long long changed = 0, sse = 0;
    write_res(a, STATS);
    p2::rows_embed<STATS>(a.v, blockIdx.x, a.v.R, gridDim.x, changed, sse);
    if (STATS)
        block_stats(changed, sse, a.res, a.slot);
}

__device__ __forceinline__ void extract_res(const P2Args &a)
{
    if (a.res && blockIdx.x == 0 && threadIdx.x == 0) {
        a.res->changed = 0;
        a.res->sse = 0;
        a.res->msg_bytes = a.v.N;
        a.res->status = STEGO_OK;
        a.res->reserved = 0;
    }
}

// A run's quarters whose vectors are in flight together in layouts that are not
// aligned (more measured slower: 5471x3647x3 12.2 us with one, 13.4 with two;
// four channels 16.6 / 15.7 us)
template <int CH>
constexpr int kQuartersAtOnce = CH == 1 ? 4 : CH == 3 ? 1 : 2;

// 5471x3647x3: 32.7 us with rows that are not whole vectors read byte by byte,
// 12.3 us as the aligned vectors around each run's pixels (one channel 18.0 ->
// 5.9, four 49.8 -> 15.8); 8192x8192x3 33.3 -> 32.9.
template <int CH>
__global__ void __launch_bounds__(512) p2_extract_units(P2Args a)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    extract_res(a);
    p2::runs_extract<CH, 4, kQuartersAtOnce<CH>>(
        a.v, (uint64_t)blockIdx.x * blockDim.x + threadIdx.x,
        p2::run_count(a.v), gridDim.x * blockDim.x);
}

__global__ void __launch_bounds__(512) p2_extract_rows(P2Args a)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    extract_res(a);
    p2::rows_extract(a.v, blockIdx.x, a.v.R, gridDim.x);
}

P2Args make_args(const uint8_t *src, uint8_t *dst, const stego_geom &g, const uint8_t *msg_in,
                 uint8_t *msg_out, uint64_t N, stego_result *res)
{
    P2Args a;
    a.v = p2::make_view(src, dst, g.width, g.height, g.channels, g.plane, msg_in, msg_out, N);
    std::memset(&a.f, 0, sizeof(a.f));
    a.res = res;
    a.slot = nullptr;
    return a;
}

int row_grid(const void *k, const Shape &sh, uint32_t rows)
{
    return persistent_grid(k, sh.threads, 0, kAnyCtas, rows ? rows : 1, 1);
}

template <bool STATS, bool INPLACE, bool SHIFTED>
const void *units_kernel(uint32_t ch)
{
    switch (ch) {
    case 1: return (const void *)p2_embed_units<1, STATS, INPLACE, SHIFTED>;
    case 3: return (const void *)p2_embed_units<3, STATS, INPLACE, SHIFTED>;
    default: return (const void *)p2_embed_units<4, STATS, INPLACE, SHIFTED>;
    }
}

// In place the units rewrite whole vectors, and only for 1, 3 or 4 channels
// with rows of whole 16-byte vectors in a 16-byte aligned buffer (the
// documented contract); elsewhere only the plane bytes are written.
bool inplace_units_ok(const uint8_t *buf, const stego_geom &g)
{
    return (((uintptr_t)buf & 15u) == 0) && g.width % 16u == 0;
}

const void *extract_units_kernel(uint32_t ch)
{
    switch (ch) {
    case 1: return (const void *)p2_extract_units<1>;
    case 3: return (const void *)p2_extract_units<3>;
    default: return (const void *)p2_extract_units<4>;
    }
}

} // namespace

// Launches the unit kernel over a.f's units.
static cudaError_t launch_units(const void *k, P2Args &a, bool stats, cudaStream_t s)
{
    const int grid = persistent_grid(k, kUnitThreads, 0, kAnyCtas, a.f.nunits,
                                     (uint64_t)kUnitThreads);
    void *args[] = {&a};
    return launch_counting(k, dim3(grid), dim3(kUnitThreads), args, 0, s, stats ? a.res : nullptr, a.slot);
}

bool p2_embed_fused(const uint8_t *cover, uint8_t *stego, const stego_geom &g,
                    const uint8_t *msg, uint64_t N, bool stats, stego_result *res,
                    cudaStream_t s, StatSlot *slot, cudaError_t *err)
{
    P2Args a = make_args(cover, stego, g, msg, nullptr, N, res);
    if (!p2::plan_units(cover, stego, (uint64_t)g.width * g.height * g.channels, g.channels,
                       g.plane, false, a.f))
        return false;
    a.slot = stats ? slot : nullptr;
    const void *k;
    if (a.f.d)
        k = stats ? units_kernel<true, false, true>(g.channels)
                  : units_kernel<false, false, true>(g.channels);
    else
        k = stats ? units_kernel<true, false, false>(g.channels)
                  : units_kernel<false, false, false>(g.channels);
    *err = launch_units(k, a, stats, s);
    return true;
}

cudaError_t p2_embed(const uint8_t *cover, uint8_t *stego, const stego_geom &g,
                     const uint8_t *msg, uint64_t N, bool stats, stego_result *res,
                     const Shape &sh, cudaStream_t s, StatSlot *slot)
{
    P2Args a = make_args(cover, stego, g, msg, nullptr, N, res);
    a.slot = stats ? slot : nullptr;
    if (cover == stego && inplace_units_ok(stego, g) &&
        p2::plan_units(cover, stego, (uint64_t)g.width * g.height * g.channels, g.channels,
                      g.plane, false, a.f)) {
        // in place over the units with carrying pixels (cut inside the
        // kernel): whole vectors instead of one byte access per plane byte
        const void *k = stats ? units_kernel<true, true, false>(g.channels)
                              : units_kernel<false, true, false>(g.channels);
        return launch_units(k, a, stats, s);
    }
    const void *k = stats ? (const void *)p2_embed_rows<true> : (const void *)p2_embed_rows<false>;
    const int grid = row_grid(k, sh, a.v.R);
    void *args[] = {&a};
    return launch_counting(k, dim3(grid), dim3(sh.threads), args, 0, s, stats ? res : nullptr, slot);
}

cudaError_t p2_extract(const uint8_t *st, const stego_geom &g, uint8_t *msg, uint64_t N,
                       stego_result *res, const Shape &sh, cudaStream_t s)
{
    P2Args a = make_args(st, nullptr, g, nullptr, msg, N, res);
    void *args[] = {&a};
    if (p2::unit_channels(g.channels)) {
        const void *k = extract_units_kernel(g.channels);
        const uint64_t runs = p2::run_count(a.v);
        const int grid = persistent_grid(k, sh.threads, 0, kAnyCtas, runs ? runs : 1,
                                         (uint64_t)sh.threads);
        return launch_dependent(k, dim3(grid), dim3(sh.threads), args, 0, s);
    }
    const void *k = (const void *)p2_extract_rows;
    const int grid = row_grid(k, sh, a.v.R);
    return launch_dependent(k, dim3(grid), dim3(sh.threads), args, 0, s);
}

} // namespace stego

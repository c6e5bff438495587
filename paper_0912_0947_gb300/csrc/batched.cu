// batched.cu -- many covers or video frames of uneven sizes in one persistent
// launch.  The paper runs its routine once per image row and per frame
// (Section VI, last paragraph; image/video frames, Section III) with a
// device allocation, two copies and a launch each time; here every cover of
// a batch is cut into fixed-size tiles that one persistent grid claims from
// a work counter.
//
// Per call, stream-ordered launches (all capturable in a CUDA graph):
//   1. prep      one thread per descriptor: validate it, (extract) read its
//                32-bit header, write its result; exclusive scan of the tile
//                counts into tile offsets, totals, work counter reset;
//   2. persist   SMs x occupancy CTAs: claim `chunk` consecutive tiles at a
//                time with one atomicAdd (the next claim is issued while the
//                current chunk is processed), find the owning descriptor by
//                a 32-way search over the offsets once per chunk, and run the
//                same per-vector code as the single-cover kernels on each
//                tile; one persistent kernel per tile space (one-bit stream
//                on 16-byte aligned buffers, one-bit stream on misaligned
//                buffers, paper layout), each exiting at once when its space
//                is empty.
// Workspace (caller-owned scratch, 16-byte aligned):
//   [0, 64)                 head: tile totals and work counters
//   [64, 64 + 24(n+1))      tile offsets of the three spaces (counts before
//                           the scan)
//   [info_off, +64n)        per-descriptor derived sizes, geometry and mode
// Both layouts batch: the one-bit stream in tiles of cover bytes; the
// paper's layout (Sections VI/VII) in tiles of 16-pixel units (1, 3 or 4
// channels) or of whole rows (copy, barrier, scatter out of place; scatter in
// place) and, for extraction, of 16-byte message runs or rows, with the
// routines the single-image kernels use.  The paper layout has its own persistent
// kernels (own tile offsets and counter), so its register needs do not
// touch the stream kernels'.
#include <cooperative_groups.h>
#include <cstring>
#include <mutex>

#include "p2_device.cuh"
#include "s1_device.cuh"

namespace stego {
namespace {

struct WsHead {
    unsigned long long total;     // one-bit stream tiles, aligned buffers
    unsigned long long counter;
    unsigned long long total_p;   // paper-layout tiles
    unsigned long long counter_p;
    unsigned long long total_m;   // one-bit stream tiles, misaligned buffers
    unsigned long long counter_m;
    unsigned long long pad[2];
};

struct DescInfo {
    uint64_t n_bytes; // stream embed: bytes written; stream extract: 8*len
    uint64_t t_bytes; // stream embed: carrying bytes; paper: R | L_last << 32
    uint64_t len;     // stream embed: stream bytes; extract / paper: message bytes
    uint32_t nbits;   // header value
    uint32_t bits;    // kHeader | kVec | kMsgEven | kFunnel
    uint32_t W, H;    // paper layout geometry; misaligned stream: head bytes,
                      // funnel byte selector
    uint32_t channels, plane; // misaligned stream embed: channels = Q (funnel word offset)
    uint32_t mode;     // paper layout: one of the kP2* work kinds
    uint32_t per_tile; // paper layout: units, rows or runs per tile
    uint32_t nunits;   // paper layout in units: their number (0: another mode)
    uint32_t flat;     // their head bytes (16 bits), cover shift and plane position
};
static_assert(sizeof(DescInfo) == 64, "DescInfo is 64 bytes");

constexpr uint32_t kHeader = 1u, kVec = 2u, kMsgEven = 4u;
// misaligned stream embed: cover and stego at different addresses mod 16
// (stego vectors joined from cover vector pairs); otherwise the same
// misalignment (vectors after a scalar head)
constexpr uint32_t kFunnel = 8u;
// paper-layout work kinds (0 = the one-bit stream layout); kP2RunsAligned: see
// p2::runs_aligned
constexpr uint32_t kP2Units = 1u, kP2RowsCopy = 2u, kP2Rows = 3u, kP2Runs = 4u, kP2RowsX = 5u,
                   kP2UnitsInPlace = 6u, kP2RunsAligned = 7u;
// Threads of the paper-layout persistent kernels' CTAs.  Unit and run tiles
// hold a whole number of CTA rounds (tile_bytes rounded down), so that no
// round runs with idle threads in the middle of a cover.
constexpr uint32_t kP2Threads = 256u;
__device__ __forceinline__ uint64_t whole_rounds(uint64_t per)
{
    return per >= kP2Threads ? per / kP2Threads * kP2Threads : per;
}
// Most tiles per claim, of the stream layout and of the paper's (see
// claim_size): long runs while there are many tiles, so that a large batch pays
// few set-ups, and single tiles where there are few, so that a small batch
// spreads over as many CTAs as there are and all end together.  kLargeChunk: of
// embeds in shapes other than the default one, whose few CTAs per SM leave the time
// between two claims in the open (1024 uneven covers, 512 threads, statistics, four
// and two vectors: 826 and 734 us with two tiles, 798 and 721 with four).
constexpr uint32_t kChunk = 2u, kPaperChunk = 4u, kLargeChunk = 4u;

// Workspace: head (64 B), aligned-stream, paper and misaligned-stream tile
// offsets (n+1 each), per-descriptor info (64 B each, 16-byte aligned).
constexpr uint64_t startp_off(uint32_t n) { return 64ull + 8ull * ((uint64_t)n + 1); }
constexpr uint64_t startm_off(uint32_t n) { return 64ull + 16ull * ((uint64_t)n + 1); }
constexpr uint64_t info_off(uint32_t n)
{
    return (64ull + 24ull * ((uint64_t)n + 1) + 15ull) & ~15ull;
}

struct WsView {
    WsHead *head;
    unsigned long long *start;   // stream-layout tile offsets, aligned buffers
    unsigned long long *start_p; // paper-layout tile offsets
    unsigned long long *start_m; // stream-layout tile offsets, misaligned buffers
    DescInfo *info;
};

WsView ws_view(void *ws, uint32_t n)
{
    WsView v;
    v.head = reinterpret_cast<WsHead *>(ws);
    v.start = reinterpret_cast<unsigned long long *>((char *)ws + 64);
    v.start_p = reinterpret_cast<unsigned long long *>((char *)ws + startp_off(n));
    v.start_m = reinterpret_cast<unsigned long long *>((char *)ws + startm_off(n));
    v.info = reinterpret_cast<DescInfo *>((char *)ws + info_off(n));
    return v;
}

__device__ __forceinline__ bool d_overlap(const void *p, uint64_t np, const void *q, uint64_t nq)
{
    if (np == 0 || nq == 0 || p == nullptr || q == nullptr)
        return false;
    const uintptr_t a = (uintptr_t)p, b = (uintptr_t)q;
    return a < b + nq && b < a + np;
}

__device__ __forceinline__ bool d_aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// ---------------------------------------------------------------------------
// 1. prep
// ---------------------------------------------------------------------------

__device__ __forceinline__ void clear_info(DescInfo &inf)
{
    inf.n_bytes = inf.t_bytes = inf.len = 0;
    inf.nbits = inf.bits = 0;
    inf.W = inf.H = inf.channels = inf.plane = 0;
    inf.mode = inf.per_tile = 0;
    inf.nunits = inf.flat = 0;
}

// Paper-layout geometry of a descriptor: channels > 0, plane < channels and
// width * height * channels == cover_bytes (Section VI step 2).
__device__ __forceinline__ bool paper_geom_ok(const stego_desc &D)
{
    const stego_geom &g = D.geom;
    return g.channels > 0 && g.plane < g.channels &&
           (uint64_t)g.width * g.height * g.channels == D.cover_bytes;
}

__device__ __forceinline__ void paper_info(const stego_desc &D, DescInfo &inf, uint64_t N)
{
    const uint32_t Q = D.geom.width / 4u;
    const uint64_t R = Q ? (N + Q - 1) / Q : 0u; // as in p2::make_view
    inf.t_bytes = R | (R ? (N - (R - 1) * Q) << 32 : 0u);
    inf.len = N;
    inf.W = D.geom.width;
    inf.H = D.geom.height;
    inf.channels = D.geom.channels;
    inf.plane = D.geom.plane;
}

// Whole rows per tile for the row-based work kinds (at least one).
__device__ __forceinline__ uint64_t rows_for(const stego_desc &D, uint32_t tile_bytes)
{
    const uint64_t rb = (uint64_t)D.geom.width * D.geom.channels;
    const uint64_t r = rb ? tile_bytes / rb : 1u;
    return r ? r : 1u;
}

// Tiles of one descriptor, or of several, in the three tile spaces: aligned
// stream, paper layout, misaligned stream.
struct Tiles {
    unsigned long long s, p, m;
};

__device__ __forceinline__ Tiles operator+(const Tiles &a, const Tiles &b)
{
    return Tiles{a.s + b.s, a.p + b.p, a.m + b.m};
}

// Validates descriptor d, writes its derived sizes and its result,
// and returns its tile count in the space of its kind.
__device__ __forceinline__ Tiles prep_embed(const stego_desc &D, uint32_t d, stego_result *results,
                                         const WsView &ws, uint32_t tile_bytes)
{
    const uint32_t layout = D.flags & STEGO_LAYOUT_MASK;
    const bool header = (D.flags & STEGO_HEADER_BE32) != 0;
    const bool inplace = D.stego == D.cover;
    int st = STEGO_OK;
    if (D.flags & ~(STEGO_LAYOUT_MASK | STEGO_HEADER_BE32 | STEGO_FUSE_STATS))
        st = STEGO_E_INVAL;
    else if (layout != STEGO_LAYOUT_STREAM1 && layout != STEGO_LAYOUT_PAPER2)
        st = STEGO_E_INVAL;
    else if (D.cover_bytes > 0 && (!D.cover || !D.stego))
        st = STEGO_E_INVAL;
    else if (D.msg_bytes > 0 && !D.msg)
        st = STEGO_E_INVAL;
    else if (!inplace && d_overlap(D.cover, D.cover_bytes, D.stego, D.cover_bytes))
        st = STEGO_E_INVAL;
    else if (d_overlap(D.msg, D.msg_bytes, D.stego, D.cover_bytes))
        st = STEGO_E_INVAL;
    else if (layout == STEGO_LAYOUT_PAPER2) {
        if (header || !paper_geom_ok(D))
            st = STEGO_E_INVAL;
        else if (D.msg_bytes > (uint64_t)(D.geom.width / 4u) * D.geom.height)
            st = STEGO_E_CAPACITY;
    } else {
        uint64_t cap = D.cover_bytes / 8u;
        if (header) {
            cap = cap >= 4u ? cap - 4u : 0u;
            if (cap > 0x1FFFFFFFull)
                cap = 0x1FFFFFFFull;
        }
        if (D.msg_bytes > cap || (header && D.cover_bytes < 32))
            st = STEGO_E_CAPACITY;
    }
    DescInfo inf;
    clear_info(inf);
    unsigned long long tiles = 0;
    bool mis = false;
    if (st == STEGO_OK && layout == STEGO_LAYOUT_PAPER2) {
        paper_info(D, inf, D.msg_bytes);
        const uint32_t ch = D.geom.channels;
        const uint64_t rows_per_tile = rows_for(D, tile_bytes);
        const p2::View v = p2::make_view(nullptr, nullptr, D.geom.width, D.geom.height, ch,
                                         D.geom.plane, nullptr, nullptr, D.msg_bytes);
        Flat f;
        const bool flat = p2::plan_units(D.cover, D.stego, D.cover_bytes, ch, D.geom.plane, true, f);
        if (flat && (!inplace || (d_aligned16(D.cover) && D.geom.width % 16u == 0))) {
            // one-pass units, for 1, 3 or 4 channels, any row length and
            // any addresses; in place (rows of whole vectors, 16-byte
            // aligned) the units with carrying pixels, written back whole
            const uint64_t units = inplace ? p2::carrying_units(v, f) : f.nunits;
            const uint64_t per =
                whole_rounds(tile_bytes / (16u * ch) ? tile_bytes / (16u * ch) : 1u);
            inf.mode = inplace ? kP2UnitsInPlace : kP2Units;
            inf.per_tile = (uint32_t)per;
            inf.n_bytes = units;
            inf.nunits = (uint32_t)f.nunits;
            inf.flat = f.h | (f.d << 16) | (f.ph << 24);
            tiles = units ? (units + per - 1) / per : 1u; // (at least the edge bytes)
        } else if (!inplace) {
            inf.mode = kP2RowsCopy;
            inf.per_tile = (uint32_t)rows_per_tile;
            tiles = (D.geom.height + rows_per_tile - 1) / rows_per_tile;
        } else {
            inf.mode = kP2Rows;
            inf.per_tile = (uint32_t)rows_per_tile;
            tiles = (v.R + rows_per_tile - 1) / rows_per_tile;
        }
    } else if (st == STEGO_OK) {
        inf.len = D.msg_bytes + (header ? 4u : 0u);
        inf.t_bytes = 8u * inf.len;
        inf.n_bytes = inplace ? inf.t_bytes : D.cover_bytes;
        inf.nbits = (uint32_t)(8u * D.msg_bytes);
        inf.bits = (header ? kHeader : 0u) |
                   ((d_aligned16(D.cover) && d_aligned16(D.stego)) ? kVec : 0u) |
                   ((((uintptr_t)D.msg & 1u) == 0) ? kMsgEven : 0u);
        tiles = (inf.n_bytes + tile_bytes - 1) / tile_bytes;
        if (!(inf.bits & kVec)) {
            // misaligned: aligned vectors after h head bytes, in tiles
            // of tile_bytes/16 vectors, when at least one vector fits
            const uint32_t hc = (uint32_t)((16u - ((uintptr_t)D.cover & 15u)) & 15u);
            const uint32_t hs = (uint32_t)((16u - ((uintptr_t)D.stego & 15u)) & 15u);
            const bool same = (((uintptr_t)D.cover ^ (uintptr_t)D.stego) & 15u) == 0;
            const uint32_t h = same ? hc : hs;
            if ((same || !inplace) && inf.n_bytes >= (uint64_t)h + 16u) {
                const uint64_t nvb = (inf.n_bytes - h) >> 4;
                const uint64_t tv = tile_bytes / 16u;
                inf.W = h;
                if (!same) {
                    const uint32_t dd = (uint32_t)(((uintptr_t)D.cover + hs) & 15u);
                    const uint32_t b = dd & 3u;
                    inf.bits |= kFunnel;
                    inf.H = b | ((b + 1) << 4) | ((b + 2) << 8) | ((b + 3) << 12);
                    inf.channels = dd >> 2;
                }
                inf.per_tile = (uint32_t)tv;
                inf.mode = 0;
                tiles = (nvb + tv - 1) / tv;
                mis = true;
            }
        }
    }
    ws.info[d] = inf;
    stego_result r;
    r.changed = 0;
    r.sse = 0;
    r.msg_bytes = st == STEGO_OK ? D.msg_bytes : 0u;
    r.status = st;
    r.reserved = 0;
    results[d] = r;
    return Tiles{inf.mode || mis ? 0ull : tiles, inf.mode ? tiles : 0ull, mis ? tiles : 0ull};
}

// Validates descriptor d, writes its derived sizes and its result (a header read),
// and returns its tile count in the space of its kind.
__device__ __forceinline__ Tiles prep_extract(const stego_desc &D, uint32_t d, stego_result *results,
                                         const WsView &ws, uint32_t tile_bytes)
{
    const uint32_t layout = D.flags & STEGO_LAYOUT_MASK;
    const bool header = (D.flags & STEGO_HEADER_BE32) != 0;
    int st = STEGO_OK;
    uint64_t len = 0;
    uint32_t nbits = 0;
    if (D.flags & ~(STEGO_LAYOUT_MASK | STEGO_HEADER_BE32 | STEGO_FUSE_STATS))
        st = STEGO_E_INVAL;
    else if (layout != STEGO_LAYOUT_STREAM1 && layout != STEGO_LAYOUT_PAPER2)
        st = STEGO_E_INVAL;
    else if (layout == STEGO_LAYOUT_PAPER2 && (header || !paper_geom_ok(D)))
        st = STEGO_E_INVAL;
    else if (D.cover_bytes > 0 && !D.cover)
        st = STEGO_E_INVAL;
    else if (D.msg_bytes > 0 && !D.msg)
        st = STEGO_E_INVAL;
    else if (d_overlap(D.msg, D.msg_bytes, D.cover, D.cover_bytes))
        st = STEGO_E_INVAL;
    else if (layout == STEGO_LAYOUT_PAPER2) {
        len = D.msg_len;
        if (len > (uint64_t)(D.geom.width / 4u) * D.geom.height)
            st = STEGO_E_CAPACITY;
        else if (len > D.msg_bytes)
            st = STEGO_E_MSG_TOO_SMALL;
    } else if (header) {
        if (D.cover_bytes < 32) {
            st = STEGO_E_BAD_HEADER;
        } else {
            if (d_aligned16(D.cover)) {
                const uint4 *h = reinterpret_cast<const uint4 *>(D.cover);
                const uint4 h0 = h[0], h1 = h[1];
                nbits = (s1::lsb16(h0) << 16) | s1::lsb16(h1);
            } else {
                for (int k = 0; k < 32; ++k)
                    nbits |= (uint32_t)(D.cover[k] & 1u) << (31 - k);
            }
            st = s1::header_status(D.cover_bytes, D.msg_bytes, nbits);
            len = nbits >> 3;
        }
    } else {
        len = D.msg_len;
        if (len > D.cover_bytes / 8u)
            st = STEGO_E_CAPACITY;
        else if (len > D.msg_bytes)
            st = STEGO_E_MSG_TOO_SMALL;
    }
    if (st != STEGO_OK)
        len = 0;
    DescInfo inf;
    clear_info(inf);
    unsigned long long tiles = 0;
    bool mis = false;
    if (layout == STEGO_LAYOUT_PAPER2 && st == STEGO_OK) {
        paper_info(D, inf, len);
        const p2::View v = p2::make_view(D.cover, nullptr, D.geom.width, D.geom.height,
                                         D.geom.channels, D.geom.plane, nullptr, D.msg, len);
        if (p2::unit_channels(D.geom.channels)) {
            const uint64_t runs = p2::run_count(v);
            const uint64_t per = whole_rounds(tile_bytes / (64u * D.geom.channels)
                                                  ? tile_bytes / (64u * D.geom.channels)
                                                  : 1u);
            inf.mode = p2::runs_aligned(v) ? kP2RunsAligned : kP2Runs;
            inf.per_tile = (uint32_t)per;
            tiles = (runs + per - 1) / per;
        } else {
            const uint64_t per = rows_for(D, tile_bytes);
            inf.mode = kP2RowsX;
            inf.per_tile = (uint32_t)per;
            tiles = (v.R + per - 1) / per;
        }
    } else {
        inf.len = len;
        inf.n_bytes = 8u * len;
        inf.nbits = nbits;
        const uint8_t *carrying = D.cover + (header ? 32u : 0u);
        inf.bits = (header ? kHeader : 0u) | (d_aligned16(carrying) ? kVec : 0u) |
                   ((((uintptr_t)D.msg & 1u) == 0) ? kMsgEven : 0u);
        tiles = (inf.n_bytes + tile_bytes - 1) / tile_bytes;
        if (!(inf.bits & kVec) && len >= 2) {
            // misaligned carrying bytes: message byte pairs from aligned
            // vector pairs, in tiles of tile_bytes/16 pairs
            const uint64_t tv = tile_bytes / 16u;
            inf.per_tile = (uint32_t)tv;
            tiles = ((len >> 1) + tv - 1) / tv;
            mis = true;
        }
    }
    ws.info[d] = inf;
    stego_result r;
    r.changed = 0;
    r.sse = 0;
    r.msg_bytes = len;
    r.status = st;
    r.reserved = 0;
    results[d] = r;
    return Tiles{inf.mode || mis ? 0ull : tiles, inf.mode ? tiles : 0ull, mis ? tiles : 0ull};
}

// Preparation of the whole batch in one launch: the descriptors are dealt in
// order to the threads of a cluster of up to eight CTAs (one CTA up to 1024
// descriptors), consecutive ones to a thread; each thread prepares its own and
// keeps their tile counts, and the exclusive scan goes through warp shuffles,
// the CTA's shared memory and the shared memory of the cluster's CTAs below.
// Bound by a chain of memory latencies (descriptor, stego header, results);
// as two launches, the scan a single CTA's 30 barriered steps over counts in
// global memory, it took 3.4-4.0 + 9 us for 16 covers.
constexpr int kPrepThreads = 1024;
constexpr uint32_t kPrepCluster = 8;

__device__ __forceinline__ Tiles shfl_up(const Tiles &v, int o)
{
    return Tiles{__shfl_up_sync(0xFFFFFFFFu, v.s, o), __shfl_up_sync(0xFFFFFFFFu, v.p, o),
                 __shfl_up_sync(0xFFFFFFFFu, v.m, o)};
}

// Inclusive scan of v over the warp.
__device__ __forceinline__ Tiles warp_scan(Tiles v, uint32_t lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Tiles u = shfl_up(v, o);
        if (lane >= (uint32_t)o)
            v = v + u;
    }
    return v;
}

template <bool EMBED>
__global__ void __launch_bounds__(kPrepThreads) prep_batch(const stego_desc *descs, uint32_t n,
                                                           stego_result *results, WsView ws,
                                                           uint32_t tile_bytes)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank(), ranks = cluster.num_blocks();
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __shared__ Tiles warp_sum[32];
    __shared__ Tiles cta_sum;
    // descriptors [b, e) are this thread's
    const uint64_t per = ((uint64_t)n + (uint64_t)ranks * blockDim.x - 1) / ((uint64_t)ranks * blockDim.x);
    const uint64_t b0 = ((uint64_t)rank * blockDim.x + threadIdx.x) * per;
    const uint32_t b = (uint32_t)(b0 < n ? b0 : n), e = (uint32_t)(b0 + per < n ? b0 + per : n);
    Tiles sum{0ull, 0ull, 0ull}; // (with one descriptor per thread its counts stay in registers)
    for (uint32_t d = b; d < e; ++d) {
        const stego_desc D = descs[d];
        const Tiles t = EMBED ? prep_embed(D, d, results, ws, tile_bytes)
                              : prep_extract(D, d, results, ws, tile_bytes);
        if (per > 1) {
            ws.start[d] = t.s;
            ws.start_p[d] = t.p;
            ws.start_m[d] = t.m;
        }
        sum = sum + t;
    }
    const Tiles incl = warp_scan(sum, lane);
    if (lane == 31)
        warp_sum[w] = incl;
    __syncthreads();
    if (w == 0) {
        const Tiles v = warp_scan(lane < nw ? warp_sum[lane] : Tiles{0ull, 0ull, 0ull}, lane);
        warp_sum[lane] = v;
        if (lane == nw - 1)
            cta_sum = v;
    }
    if (ranks > 1)
        cluster.sync(); // every CTA's sum is there (and this CTA's warp sums)
    else
        __syncthreads();
    Tiles run{incl.s - sum.s, incl.p - sum.p, incl.m - sum.m};
    if (w)
        run = run + warp_sum[w - 1];
    for (uint32_t r = 0; r < rank; ++r)
        run = run + *cluster.map_shared_rank(&cta_sum, r);
    for (uint32_t d = b; d < e; ++d) {
        Tiles t = sum;
        if (per > 1)
            t = Tiles{ws.start[d], ws.start_p[d], ws.start_m[d]};
        ws.start[d] = run.s;
        ws.start_p[d] = run.p;
        ws.start_m[d] = run.m;
        run = run + t;
    }
    if (rank == ranks - 1 && threadIdx.x == blockDim.x - 1) { // the last in order: the totals
        ws.start[n] = run.s;
        ws.start_p[n] = run.p;
        ws.start_m[n] = run.m;
        ws.head->total = run.s;
        ws.head->counter = 0;
        ws.head->total_p = run.p;
        ws.head->counter_p = 0;
        ws.head->total_m = run.m;
        ws.head->counter_m = 0;
    }
    if (ranks > 1)
        cluster.sync(); // the sums stay until the CTAs above have read them
}

// ---------------------------------------------------------------------------
// 2. persistent kernels
// ---------------------------------------------------------------------------

// Largest d < n with start[d] <= t (start[0] = 0 <= t < start[n]), by whole
// warps (CTAs are of whole warps) with the same arguments: 32 places are looked
// up at once, two dependent loads up to 1024 covers where halving took ten,
// all of them on the CTA's path between two claims.  Per call, device time,
// halving against this: 256 covers of sides 64 to 512 embed 24.4 -> 23.0 us,
// extract 19.0 -> 16.7; 4096 uneven covers embed 2459 -> 2441; 1024 paper covers
// 900 -> 896 and 392 -> 388; 300 HD paper frames extract 190 -> 188 (all before the
// paper kernels found rows by divisions).
__device__ __forceinline__ uint32_t owner_of(const unsigned long long *start, uint32_t n,
                                             unsigned long long t)
{
    uint32_t lo = 0, m = n; // start[lo] <= t < start[lo + m]
    while (m > 1) {
        const uint32_t step = (m - 1) / 32u + 1u;
        const uint32_t at = ((threadIdx.x & 31u) + 1u) * step;
        const uint32_t c = __popc(__ballot_sync(~0u, at < m && start[lo + at] <= t));
        lo += c * step;
        m = m - c * step < step ? m - c * step : step;
    }
    return lo;
}

// Warp-level flush of per-thread statistics into one descriptor's result.
__device__ __forceinline__ void flush_stats(unsigned long long &changed, unsigned long long &sse,
                                            stego_result *res)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        changed += __shfl_down_sync(0xFFFFFFFFu, changed, o);
        sse += __shfl_down_sync(0xFFFFFFFFu, sse, o);
    }
    if ((threadIdx.x & 31u) == 0 && res) {
        if (changed)
            atomicAdd(reinterpret_cast<unsigned long long *>(&res->changed), changed);
        if (sse)
            atomicAdd(reinterpret_cast<unsigned long long *>(&res->sse), sse);
    }
    changed = 0;
    sse = 0;
}

// Tiles of a claim: a quarter of the CTA's share of `left` tiles, at most MAX.
template <uint32_t MAX>
__device__ __forceinline__ uint32_t claim_size(unsigned long long left)
{
    const uint32_t n = (left >> 32) ? MAX : (uint32_t)left / (4u * gridDim.x);
    return n < 1u ? 1u : n < MAX ? n : MAX;
}

// Tiles of a small batch are cut in 2^shift parts (down to 4096 bytes), until
// every CTA has a few or they are no smaller than that: 16 covers of sides 64
// to 512 are 50 tiles of 64 KiB, which 50 CTAs took one after another.  A part
// is a whole number of 16-byte vectors, so that the parts of tile_bytes (and of
// a misaligned tile's tile_bytes / 16 vectors or byte pairs) make up the tile.
__device__ __forceinline__ uint32_t split_shift(unsigned long long total, uint32_t tile_bytes)
{
    uint32_t s = 0;
    while (total << s < 2ull * gridDim.x && (tile_bytes >> (s + 1)) >= 4096u &&
           (tile_bytes & ((32u << s) - 1u)) == 0u)
        ++s;
    return s;
}

// The claim loop shared by both directions, over `total` tiles, each in 2^shift
// parts: calls body for the parts of the chunks this CTA claims, in order.  MERGE:
// body(d, first, count) once for every run of `count` consecutive tiles of one
// descriptor, one set-up for all of them (a call per tile cost the paper layout's
// kernels as many instructions as a round of their threads); parts of a tile, and
// the stream kernels' tiles, singly: body(d, first) (their set-up is a few loads,
// and merged ranges cost persist_embed<4, true> two registers and with them the
// third CTA per SM).  `first` counts the descriptor's parts.
template <bool MERGE, uint32_t MAX, typename Body>
__device__ __forceinline__ void claim_loop(const unsigned long long *start,
                                           unsigned long long total, uint32_t shift,
                                           unsigned long long *counter, uint32_t n, Body &&body)
{
    __shared__ unsigned long long s_claim;
    __shared__ uint32_t s_count;
    const unsigned long long parts = total << shift;
    if (threadIdx.x == 0 && total) {
        const uint32_t cnt = claim_size<MAX>(parts);
        s_count = cnt;
        s_claim = atomicAdd(counter, (unsigned long long)cnt);
    }
    if (!total)
        return;
    __syncthreads();
    for (;;) {
        const unsigned long long c0 = s_claim, ce = c0 + s_count;
        __syncthreads(); // every thread has read the claim
        if (c0 >= parts)
            break;
        const unsigned long long c1 = ce < parts ? ce : parts;
        // before the claim: warp 0 would enter the search only when its atomic is
        // back (16 covers, extract: 10.7 us with the search after it, 9.9 so)
        uint32_t d = owner_of(start, n, c0 >> shift);
        if (threadIdx.x == 0) { // next claim in flight while this chunk runs
            const uint32_t cnt = claim_size<MAX>(parts - c1);
            s_count = cnt;
            s_claim = atomicAdd(counter, (unsigned long long)cnt);
        }
        unsigned long long t = c0;
        while (t < c1) {
            while (start[d + 1] <= t >> shift)
                ++d;
            const unsigned long long first = t - (start[d] << shift);
            if constexpr (MERGE) {
                uint32_t cnt = 1;
                if (shift == 0)
                    cnt = (uint32_t)((start[d + 1] < c1 ? start[d + 1] : c1) - t);
                t += cnt;
                body(d, first, cnt);
            } else {
                ++t;
                body(d, first);
            }
        }
        __syncthreads(); // the next claim is visible
    }
}

// What the CTA's threads need to know of a paper-layout cover, in shared memory:
// read where it is used, it costs the routines below no registers (passed by
// value it lay on each thread's stack, and a quarter of the instructions
// were its loads and stores).
struct PaperJob {
    p2::View v;
    Flat f;
};

__device__ __forceinline__ const PaperJob &paper_job(const stego_desc &D, const DescInfo &inf,
                                                     bool embed)
{
    __shared__ PaperJob job;
    __syncthreads(); // every thread is done with the previous cover
    if (threadIdx.x == 0) {
        p2::View &v = job.v;
        v.src = D.cover;
        v.dst = embed ? D.stego : nullptr;
        v.msg_in = embed ? D.msg : nullptr;
        v.msg_out = embed ? nullptr : D.msg;
        v.N = inf.len;
        v.W = inf.W;
        v.H = inf.H;
        v.channels = inf.channels;
        v.plane = inf.plane;
        v.Q = inf.W / 4u;
        v.R = (uint32_t)inf.t_bytes;
        v.L_last = (uint32_t)(inf.t_bytes >> 32);
        v.kmul = 4u;
        job.f.h = inf.flat & 0xFFFFu;
        job.f.d = (inf.flat >> 16) & 0xFFu;
        job.f.ph = inf.flat >> 24;
        job.f.x0 = inf.channels == 1 ? job.f.h
                                     : (job.f.h + job.f.ph - inf.plane) / inf.channels;
        job.f.nunits = inf.nunits;
        job.f.sel = make_sel(inf.channels, job.f.ph);
    }
    __syncthreads();
    return job;
}

// Units, rows or runs [b0, b1) of tiles lt .. lt + cnt - 1, or of part lt.
__device__ __forceinline__ void paper_part(const DescInfo &inf, unsigned long long lt, uint32_t cnt,
                                           uint32_t shift, uint64_t &b0, uint64_t &b1)
{
    const uint64_t tile = (lt >> shift) * inf.per_tile;
    const uint32_t per = (inf.per_tile + (1u << shift) - 1) >> shift; // of a part
    const uint32_t at = (uint32_t)(lt & ((1u << shift) - 1)) * per;
    b0 = tile + (at < inf.per_tile ? at : inf.per_tile);
    b1 = shift ? tile + (at + per < inf.per_tile ? at + per : inf.per_tile)
               : b0 + (uint64_t)cnt * inf.per_tile;
}

// Tiles lt .. lt + cnt - 1 of a paper-layout cover (the CTA's threads together).
template <bool STATS>
__device__ __forceinline__ void paper_embed_tile(const stego_desc &D, const DescInfo &inf,
                                                 unsigned long long lt, uint32_t cnt,
                                                 uint32_t shift, unsigned long long &changed,
                                                 unsigned long long &sse)
{
    const PaperJob &job = paper_job(D, inf, true);
    uint64_t b0, b1;
    paper_part(inf, lt, cnt, shift, b0, b1);
    if (inf.mode == kP2Units || inf.mode == kP2UnitsInPlace) {
        // in place the same code runs over the carrying rows' units only:
        // each unit is read and written back by one thread, so src == dst is
        // safe, and the last row's units past its carrying columns are
        // rewritten unchanged (one instantiation keeps the registers down)
        if (b0 >= b1 || (b0 >= inf.n_bytes && lt != 0))
            return; // a part past the tile's or the cover's end
        const uint32_t k0 = (uint32_t)b0 + threadIdx.x;
        const uint32_t k1 = (uint32_t)(b1 < inf.n_bytes ? b1 : inf.n_bytes);
        // one unit per thread, loaded by the thread itself: when these kernels
        // had 80 registers and three CTAs per SM, a form staged through shared
        // memory spilled more and ran slower (600 video frames: 1.53 against
        // 1.26 ms), and so did the cp.async pipeline of the single-cover kernel
        // (1.34-1.83 ms; 256 large RGB covers at 64 registers 3187 against 2545 us)
        switch (inf.channels) {
        case 1: p2::units_embed<1, STATS, false, true>(job.v, job.f, k0, k1, blockDim.x, changed, sse); break;
        case 3: p2::units_embed<3, STATS, false, true>(job.v, job.f, k0, k1, blockDim.x, changed, sse); break;
        default: p2::units_embed<4, STATS, false, true>(job.v, job.f, k0, k1, blockDim.x, changed, sse); break;
        }
        if (b0 == 0 || b1 >= inf.n_bytes)
            p2::edge_bytes<STATS>(job.v, job.f, b0 == 0, b1 >= inf.n_bytes, changed, sse);
        return;
    }
    const uint32_t r0 = (uint32_t)b0;
    const uint32_t r1 = (uint32_t)(b1 < inf.H ? b1 : inf.H);
    if (inf.mode == kP2RowsCopy) {
        p2::rows_copy(job.v, r0, r1);
        __syncthreads(); // the copy lands before the scatter overwrites plane bytes
    }
    p2::rows_embed<STATS>(job.v, r0, r1, 1, changed, sse);
}

// a run's quarters whose vectors are in flight together, in aligned layouts
// and others
constexpr int kBatchAligned = 2, kBatchQuarters = 1;

__device__ __forceinline__ void paper_extract_tile(const stego_desc &D, const DescInfo &inf,
                                                   unsigned long long lt, uint32_t cnt,
                                                 uint32_t shift)
{
    uint64_t b0, b1;
    paper_part(inf, lt, cnt, shift, b0, b1);
    if (inf.mode == kP2RunsAligned) {
        // the full rows need so little of the cover that each thread reads it for
        // itself: without the barriers around paper_job, 300 HD frames 188 -> 176 us
        p2::View v;
        v.src = D.cover;
        v.msg_out = D.msg;
        v.W = inf.W;
        v.Q = inf.W / 4u;
        v.plane = inf.plane;
        v.R = (uint32_t)inf.t_bytes;
        v.L_last = (uint32_t)(inf.t_bytes >> 32);
        const uint64_t full = p2::aligned_full_runs(v), ke = b1 < full ? b1 : full;
        switch (inf.channels) {
        case 1: p2::aligned_runs<1, 4, true>(v, b0 + threadIdx.x, ke, blockDim.x); break;
        case 3: p2::aligned_runs<3, kBatchAligned, true>(v, b0 + threadIdx.x, ke, blockDim.x); break;
        default: p2::aligned_runs<4, kBatchAligned, true>(v, b0 + threadIdx.x, ke, blockDim.x); break;
        }
        if (b1 <= full || v.L_last == v.Q)
            return;
        b0 = b0 > full ? b0 : full; // the last row's
    }
    const PaperJob &job = paper_job(D, inf, false);
    if (inf.mode == kP2Runs || inf.mode == kP2RunsAligned) {
        const uint64_t runs = p2::run_count(job.v);
        const uint64_t k0 = b0 + threadIdx.x, k1 = b1 < runs ? b1 : runs;
        switch (inf.channels) {
        case 1: p2::other_runs<1, 1, true>(job.v, k0, k1, blockDim.x); break;
        case 3: p2::other_runs<3, kBatchQuarters, true>(job.v, k0, k1, blockDim.x); break;
        default: p2::other_runs<4, kBatchQuarters, true>(job.v, k0, k1, blockDim.x); break;
        }
    } else {
        p2::rows_extract(job.v, (uint32_t)b0, (uint32_t)(b1 < job.v.R ? b1 : job.v.R), 1);
    }
}

// Four vectors per thread in CTAs of at most 256 threads (the default shape)
// keep 80 registers, three CTAs per SM: 82 cost 13% of the uneven batch.  No bound
// for the others: with one CTA per SM as theirs the compiler took 56-91 registers
// in place of 32-82 (1024 uneven covers, 512 threads, no statistics, four vectors
// 794 us, so 654; with statistics, two vectors 1011, so 721).
template <int V, bool STATS, bool SMALL>
__global__ void __launch_bounds__(SMALL ? 256 : 512, SMALL ? 3 : 0) persist_embed(const stego_desc *descs, uint32_t n,
                                                     stego_result *results, WsView ws,
                                                     uint32_t tile_bytes)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    unsigned long long changed = 0, sse = 0;
    uint32_t stat_d = 0xFFFFFFFFu;
    const unsigned long long total = ws.head->total;
    const uint32_t shift = split_shift(total, tile_bytes), part_bytes = tile_bytes >> shift;
    claim_loop<false, SMALL ? kChunk : kLargeChunk>(ws.start, total, shift, &ws.head->counter, n,
               [&](uint32_t d, unsigned long long lt) {
        if (STATS && d != stat_d) {
            flush_stats(changed, sse, stat_d < n ? results + stat_d : nullptr);
            stat_d = d;
        }
        const stego_desc &D = descs[d];
        const DescInfo inf = ws.info[d];
        s1::EmbedView a;
        a.cover = D.cover;
        a.stego = D.stego;
        a.msg = D.msg;
        a.n_bytes = inf.n_bytes;
        a.t_bytes = inf.t_bytes;
        a.slen = inf.len;
        a.header = (inf.bits & kHeader) ? 1u : 0u;
        a.nbits = inf.nbits;
        a.msg_even = (inf.bits & kMsgEven) ? 1u : 0u;
        a.pad = 0;
        const uint64_t b0 = lt * part_bytes, be = b0 + part_bytes;
        const uint64_t b1 = be < inf.n_bytes ? be : inf.n_bytes;
        if (b0 >= b1)
            return; // a part past the cover's end
        if (inf.bits & kVec) {
            s1::embed_vec_range<V, STATS>(a, (b0 >> 4) + threadIdx.x, b1 >> 4,
                                          (uint64_t)blockDim.x * V, changed, sse);
            if (b1 == inf.n_bytes)
                s1::embed_tail<STATS>(a, changed, sse);
        } else {
            s1::embed_bytes_range<STATS>(a, (b0 >> 3) + threadIdx.x, (b1 + 7) >> 3, blockDim.x,
                                         changed, sse);
        }
    });
    if (STATS)
        flush_stats(changed, sse, stat_d < n ? results + stat_d : nullptr);
}

template <int V>
__global__ void __launch_bounds__(512) persist_extract(const stego_desc *descs, uint32_t n,
                                                       WsView ws, uint32_t tile_bytes)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    const unsigned long long total = ws.head->total;
    const uint32_t shift = split_shift(total, tile_bytes), part_bytes = tile_bytes >> shift;
    claim_loop<false, kChunk>(ws.start, total, shift, &ws.head->counter, n,
               [&](uint32_t d, unsigned long long lt) {
        const stego_desc &D = descs[d];
        const DescInfo inf = ws.info[d];
        s1::ExtractView x;
        x.st = D.cover;
        x.msg = D.msg;
        x.len = inf.len;
        x.base = (inf.bits & kHeader) ? 32u : 0u;
        x.msg_even = (inf.bits & kMsgEven) ? 1u : 0u;
        x.pad = 0;
        const uint64_t b0 = lt * part_bytes, be = b0 + part_bytes;
        const uint64_t b1 = be < inf.n_bytes ? be : inf.n_bytes;
        if (b0 >= b1)
            return; // a part past the cover's end
        if (inf.bits & kVec) {
            s1::extract_vec_range<V>(x, (b0 >> 4) + threadIdx.x, b1 >> 4, (uint64_t)blockDim.x * V);
            if (b1 == inf.n_bytes && (x.len & 1u) && threadIdx.x == 0)
                s1::extract_one(x, x.len - 1);
        } else {
            s1::extract_bytes_range(x, (b0 >> 3) + threadIdx.x, b1 >> 3, blockDim.x);
        }
    });
}

// One-bit stream covers whose buffers are not 16-byte aligned, in their own
// tile space and kernels, so that the aligned kernels keep their register
// budget (calling these routines from them raised persist_embed<4, true>
// from 80 to 94 registers and persist_extract<4> from 39 to 64).  A tile is
// per_tile aligned stego vectors (embed) or message byte pairs (extract);
// the routines are the single-cover kernels' (same misalignment: vectors
// after a scalar head, two per thread and round; different misalignments:
// each stego vector joined from the two aligned cover vectors around its
// bytes, the second passed from the next lane, blocks of 4 x 32 vectors per
// warp; extraction: aligned stego vectors reduced to their LSBs, a pair's
// bits cut from two lanes', four per thread).
constexpr int kMisV = 2, kMisFunnelV = 4, kMisXV = 4;

template <int Q, bool STATS>
__device__ __forceinline__ void mis_funnel(const s1::EmbedView &a, uint32_t h, uint32_t sel,
                                           uint64_t j0, uint64_t j1, unsigned long long &changed,
                                           unsigned long long &sse)
{
    s1::embed_funnel_warp<Q, STATS, kMisFunnelV>(a, h, sel, j0, j1, threadIdx.x >> 5,
                                                 blockDim.x >> 5, changed, sse);
}

// Part lt of a misaligned stream cover (the CTA's threads together).
template <bool STATS>
__device__ __forceinline__ void mis_embed_tile(const stego_desc &D, const DescInfo &inf,
                                               unsigned long long lt, uint32_t shift,
                                               unsigned long long &changed,
                                               unsigned long long &sse)
{
        s1::EmbedView a;
        a.cover = D.cover;
        a.stego = D.stego;
        a.msg = D.msg;
        a.n_bytes = inf.n_bytes;
        a.t_bytes = inf.t_bytes;
        a.slen = inf.len;
        a.header = (inf.bits & kHeader) ? 1u : 0u;
        a.nbits = inf.nbits;
        a.msg_even = (inf.bits & kMsgEven) ? 1u : 0u;
        a.pad = 0;
        const uint32_t h = inf.W;
        const uint64_t nvb = (inf.n_bytes - h) >> 4;
        // (a misaligned tile is tile_bytes / 16 vectors: whole parts, see split_shift)
        const uint64_t per = inf.per_tile >> shift;
        const uint64_t j0 = lt * per, je = j0 + per;
        const uint64_t j1 = je < nvb ? je : nvb;
        if (j0 >= j1)
            return; // a part past the cover's end
        if (inf.bits & kFunnel) {
            switch (inf.channels) {
            case 0: mis_funnel<0, STATS>(a, h, inf.H, j0, j1, changed, sse); break;
            case 1: mis_funnel<1, STATS>(a, h, inf.H, j0, j1, changed, sse); break;
            case 2: mis_funnel<2, STATS>(a, h, inf.H, j0, j1, changed, sse); break;
            default: mis_funnel<3, STATS>(a, h, inf.H, j0, j1, changed, sse); break;
            }
        } else {
            s1::embed_shift_range<kMisV, STATS>(a, h, j0 + threadIdx.x, j1,
                                                (uint64_t)blockDim.x * kMisV, changed, sse);
        }
        // the h head bytes with the first tile, the tail (under one vector)
        // with the last, one byte per thread
        const uint32_t tail = (uint32_t)(inf.n_bytes - h - (nvb << 4));
        uint64_t k = ~0ull;
        if (lt == 0 && threadIdx.x < h)
            k = threadIdx.x;
        else if (j1 == nvb && threadIdx.x >= 16 && threadIdx.x - 16 < tail)
            k = h + (nvb << 4) + (threadIdx.x - 16);
        if (k != ~0ull) {
            const uint32_t sb = k < a.t_bytes ? s1::stream_byte(a, k >> 3) : 0u;
            s1::embed_one<STATS>(a, k, sb, changed, sse);
        }
}

__device__ __forceinline__ void mis_extract_tile(const stego_desc &D, const DescInfo &inf,
                                                 unsigned long long lt, uint32_t shift)
{
        s1::ExtractView x;
        x.st = D.cover;
        x.msg = D.msg;
        x.len = inf.len;
        x.base = (inf.bits & kHeader) ? 32u : 0u;
        x.msg_even = (inf.bits & kMsgEven) ? 1u : 0u;
        x.pad = 0;
        const uint64_t np = inf.len >> 1;
        const uint64_t per = inf.per_tile >> shift;
        const uint64_t p0 = lt * per, pe = p0 + per;
        const uint64_t p1 = pe < np ? pe : np;
        if (p0 >= p1)
            return; // a part past the message's end
        s1::extract_shift_lsb<kMisXV>(x, D.cover_bytes, p0, p1, threadIdx.x >> 5,
                                      blockDim.x >> 5);
        if (p1 == np && (x.len & 1u) && threadIdx.x == 0)
            s1::extract_one(x, x.len - 1);
}

// The misaligned stream tiles' own persistent kernels, with register
// budgets of their own (inside the paper layout's kernel the embed ran at
// 0.69 of the HBM peak on 4096 covers).  The embed runs three CTAs of 256
// threads per SM at 80 registers: with one cover load per stego vector
// (the funnel's second vector shuffled from the next lane) four vectors per
// lane fit, 48 KiB of cover in flight per SM; on the 4096-cover batch at
// offsets 1..15 that took the embed from 2.95 to 2.67 ms (0.83 to 0.92 of
// the peak; the two-load form at two vectors: two CTAs of 512 threads at
// 64 registers; the shuffled form at two vectors or at four in two CTAs of
// 512 threads: 2.92-2.97 ms).  The extract runs CTAs of 128 threads (48
// registers, ten per SM), a 64 KiB tile being eight rounds of their warps:
// on the same batch 0.84 ms with 256 threads, 0.75 ms with 128, as fast as
// the aligned batch in the same launch shape (512 threads: 0.87 against
// 0.76 of the peak with 256; eight vectors per lane: 0.75-0.77 ms).
constexpr int kMisEmbedThreads = 256, kMisEmbedMinCtas = 3, kMisExtractThreads = 128;
template <bool STATS>
__global__ void __launch_bounds__(kMisEmbedThreads, kMisEmbedMinCtas)
    persist_mis_embed(const stego_desc *descs, uint32_t n, stego_result *results, WsView ws,
                      uint32_t tile_bytes)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    unsigned long long changed = 0, sse = 0;
    uint32_t stat_d = 0xFFFFFFFFu;
    const unsigned long long total = ws.head->total_m;
    const uint32_t shift = split_shift(total, tile_bytes);
    claim_loop<false, kChunk>(ws.start_m, total, shift, &ws.head->counter_m, n,
               [&](uint32_t d, unsigned long long lt) {
        if (STATS && d != stat_d) {
            flush_stats(changed, sse, stat_d < n ? results + stat_d : nullptr);
            stat_d = d;
        }
        mis_embed_tile<STATS>(descs[d], ws.info[d], lt, shift, changed, sse);
    });
    if (STATS)
        flush_stats(changed, sse, stat_d < n ? results + stat_d : nullptr);
}

__global__ void __launch_bounds__(kMisExtractThreads)
    persist_mis_extract(const stego_desc *descs, uint32_t n, WsView ws,
                      uint32_t tile_bytes)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    const unsigned long long total = ws.head->total_m;
    const uint32_t shift = split_shift(total, tile_bytes);
    claim_loop<false, kChunk>(ws.start_m, total, shift, &ws.head->counter_m, n,
               [&](uint32_t d, unsigned long long lt) {
        mis_extract_tile(descs[d], ws.info[d], lt, shift);
    });
}

// The paper layout's own persistent kernels (a separate register budget from
// the stream kernels): tiles of units, rows or runs, claimed like above.
// Capped at 64 registers for four CTAs per SM (1024 covers of sides 64 to 4096,
// half RGB: embed 960 us against 1023 with three CTAs at 80 registers, 1107
// with two, although it spills; extract of 300 frames 854 wide 105 against 114, of
// the covers 379 against 364).  One unit or run at a
// time: with four CTAs the warps hide the latency, and two in flight were
// slower.  With rows that are not whole vectors copied and then scattered byte
// by byte the same batch took 2823 us (embed) and 505 us (extract), now 893
// and 371; large RGB covers run at 0.75 of the copy rate, gray ones, with
// three times the units per byte, at 0.53.
template <bool STATS>
__global__ void __launch_bounds__(kP2Threads, 4) persist_p2_embed(const stego_desc *descs, uint32_t n,
                                                        stego_result *results, WsView ws,
                                                        uint32_t tile_bytes)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    unsigned long long changed = 0, sse = 0;
    uint32_t stat_d = 0xFFFFFFFFu;
    const unsigned long long total = ws.head->total_p;
    const uint32_t shift = split_shift(total, tile_bytes);
    claim_loop<true, kPaperChunk>(ws.start_p, total, shift, &ws.head->counter_p, n,
               [&](uint32_t d, unsigned long long lt, uint32_t cnt) {
        if (STATS && d != stat_d) {
            flush_stats(changed, sse, stat_d < n ? results + stat_d : nullptr);
            stat_d = d;
        }
        paper_embed_tile<STATS>(descs[d], ws.info[d], lt, cnt, shift, changed, sse);
    });
    if (STATS)
        flush_stats(changed, sse, stat_d < n ? results + stat_d : nullptr);
}

__global__ void __launch_bounds__(kP2Threads, 4) persist_p2_extract(const stego_desc *descs, uint32_t n,
                                                          WsView ws, uint32_t tile_bytes)
{
    grid_dependency_wait(); // launched dependent: nothing is touched before
    allow_dependents();
    const unsigned long long total = ws.head->total_p;
    const uint32_t shift = split_shift(total, tile_bytes);
    claim_loop<true, kPaperChunk>(ws.start_p, total, shift, &ws.head->counter_p, n,
               [&](uint32_t d, unsigned long long lt, uint32_t cnt) {
        paper_extract_tile(descs[d], ws.info[d], lt, cnt, shift);
    });
}

template <bool EMBED>
const void *persist_kernel(int vec, int threads, bool stats)
{
    if (EMBED) {
        switch (vec) {
        case 1: return stats ? (const void *)persist_embed<1, true, false> : (const void *)persist_embed<1, false, false>;
        case 2: return stats ? (const void *)persist_embed<2, true, false> : (const void *)persist_embed<2, false, false>;
        case 8: return stats ? (const void *)persist_embed<8, true, false> : (const void *)persist_embed<8, false, false>;
        default:
            if (threads <= 256)
                return stats ? (const void *)persist_embed<4, true, true> : (const void *)persist_embed<4, false, true>;
            return stats ? (const void *)persist_embed<4, true, false> : (const void *)persist_embed<4, false, false>;
        }
    }
    switch (vec) {
    case 1: return (const void *)persist_extract<1>;
    case 2: return (const void *)persist_extract<2>;
    case 8: return (const void *)persist_extract<8>;
    default: return (const void *)persist_extract<4>;
    }
}

uint64_t workspace_bytes(uint32_t n) { return info_off(n) + sizeof(DescInfo) * (uint64_t)n; }

template <bool EMBED>
int batched(const stego_desc *d_descs, uint32_t n, stego_result *d_results, uint32_t flags,
            const stego_tune *tune, void *d_ws, uint64_t ws_bytes, void *stream)
{
    if (flags & ~(uint32_t)STEGO_FUSE_STATS)
        return STEGO_E_INVAL;
    if (!EMBED && (flags & STEGO_FUSE_STATS))
        return STEGO_E_INVAL;
    if (tune && !tune_ok(tune))
        return STEGO_E_INVAL;
    if (n == 0)
        return STEGO_OK;
    if (!d_descs || !d_results || !d_ws)
        return STEGO_E_INVAL;
    if (((uintptr_t)d_descs & 7u) || ((uintptr_t)d_results & 7u) || ((uintptr_t)d_ws & 15u))
        return STEGO_E_INVAL;
    if (ws_bytes < workspace_bytes(n))
        return STEGO_E_NOMEM;
    cudaStream_t s = (cudaStream_t)stream;
    const Shape sh = shape_for(EMBED ? STEGO_OP_EMBED_BATCHED : STEGO_OP_EXTRACT_BATCHED, tune);
    const uint32_t tile = sh.tile_bytes;
    WsView ws = ws_view(d_ws, n);

    cudaError_t e;
    {
        // one CTA of whole warps up to kPrepThreads descriptors, then a cluster
        const uint32_t want = (n + kPrepThreads - 1) / kPrepThreads;
        uint32_t ctas = 1;
        while (ctas < want && ctas < kPrepCluster)
            ctas *= 2;
        const uint32_t threads = n < kPrepThreads ? (n + 31u) / 32u * 32u : kPrepThreads;
        uint32_t tile_arg = tile;
        void *args[] = {(void *)&d_descs, &n, &d_results, &ws, &tile_arg};
        e = launch_dependent(EMBED ? (const void *)prep_batch<true> : (const void *)prep_batch<false>,
                             dim3(ctas), dim3(threads), args, 0, s, ctas);
    }
    if (e != cudaSuccess)
        return STEGO_E_CUDA;

    const bool stats = (flags & STEGO_FUSE_STATS) != 0;
    const void *k = persist_kernel<EMBED>(sh.vec, sh.threads, stats);
    // the tile count lives on the device: launch the full persistent grid
    const int grid = persistent_grid(k, sh.threads, 0, sh.ctas_per_sm, ~0ull >> 1, 1);
    if (EMBED) {
        void *args[] = {(void *)&d_descs, &n, &d_results, &ws, (void *)&tile};
        e = launch_dependent(k, dim3(grid), dim3(sh.threads), args, 0, s);
    } else {
        void *args[] = {(void *)&d_descs, &n, &ws, (void *)&tile};
        e = launch_dependent(k, dim3(grid), dim3(sh.threads), args, 0, s);
    }
    if (e != cudaSuccess)
        return STEGO_E_CUDA;
    // misaligned stream tiles (count on the device; an empty set exits at once)
    {
        const int mis_threads = EMBED ? kMisEmbedThreads : kMisExtractThreads;
        const void *km = EMBED ? (stats ? (const void *)persist_mis_embed<true>
                                        : (const void *)persist_mis_embed<false>)
                               : (const void *)persist_mis_extract;
        const int gridm = persistent_grid(km, mis_threads, 0, 0, ~0ull >> 1, 1);
        if (EMBED) {
            void *args[] = {(void *)&d_descs, &n, &d_results, &ws, (void *)&tile};
            e = launch_dependent(km, dim3(gridm), dim3(mis_threads), args, 0, s);
        } else {
            void *args[] = {(void *)&d_descs, &n, &ws, (void *)&tile};
            e = launch_dependent(km, dim3(gridm), dim3(mis_threads), args, 0, s);
        }
    }
    if (e != cudaSuccess)
        return STEGO_E_CUDA;
    // paper-layout tiles (their count is on the device; an empty set exits at once)
    const int p2_threads = (int)kP2Threads;
    const void *kp = EMBED ? (stats ? (const void *)persist_p2_embed<true>
                                    : (const void *)persist_p2_embed<false>)
                           : (const void *)persist_p2_extract;
    const int gridp = persistent_grid(kp, p2_threads, 0, 0, ~0ull >> 1, 1);
    if (EMBED) {
        void *args[] = {(void *)&d_descs, &n, &d_results, &ws, (void *)&tile};
        e = launch_dependent(kp, dim3(gridp), dim3(p2_threads), args, 0, s);
    } else {
        void *args[] = {(void *)&d_descs, &n, &ws, (void *)&tile};
        e = launch_dependent(kp, dim3(gridp), dim3(p2_threads), args, 0, s);
    }
    return e == cudaSuccess ? STEGO_OK : STEGO_E_CUDA;
}

} // namespace
} // namespace stego

using namespace stego;

struct stego_graph {
    cudaGraph_t graph;
    cudaGraphExec_t exec;
};

extern "C" {

uint64_t stego_batched_workspace_bytes(uint32_t n) { return workspace_bytes(n); }

int stego_embed_batched(const stego_desc *d_descs, uint32_t n, stego_result *d_results,
                        uint32_t flags, const stego_tune *tune, void *d_ws, uint64_t ws_bytes,
                        void *stream)
{
    stego::Trace trace_("stego_embed_batched");
    return batched<true>(d_descs, n, d_results, flags, tune, d_ws, ws_bytes, stream);
}

int stego_extract_batched(const stego_desc *d_descs, uint32_t n, stego_result *d_results,
                          uint32_t flags, const stego_tune *tune, void *d_ws, uint64_t ws_bytes,
                          void *stream)
{
    stego::Trace trace_("stego_extract_batched");
    return batched<false>(d_descs, n, d_results, flags, tune, d_ws, ws_bytes, stream);
}

int stego_graph_capture_batched(int op, const stego_desc *d_descs, uint32_t n,
                                stego_result *d_results, uint32_t flags, const stego_tune *tune,
                                void *d_ws, uint64_t ws_bytes, stego_graph **out)
{
    stego::Trace trace_("stego_graph_capture_batched");
    if (!out || (op != STEGO_OP_EMBED_BATCHED && op != STEGO_OP_EXTRACT_BATCHED))
        return STEGO_E_INVAL;
    *out = nullptr;
    cudaStream_t s = nullptr;
    if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess)
        return STEGO_E_CUDA;
    int st = STEGO_OK;
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        cudaStreamDestroy(s);
        return STEGO_E_CUDA;
    }
    if (op == STEGO_OP_EMBED_BATCHED)
        st = stego_embed_batched(d_descs, n, d_results, flags, tune, d_ws, ws_bytes, s);
    else
        st = stego_extract_batched(d_descs, n, d_results, flags, tune, d_ws, ws_bytes, s);
    const cudaError_t ee = cudaStreamEndCapture(s, &g);
    cudaStreamDestroy(s);
    if (st != STEGO_OK) {
        if (g)
            cudaGraphDestroy(g);
        return st;
    }
    if (ee != cudaSuccess || !g)
        return STEGO_E_CUDA;
    cudaGraphExec_t ex = nullptr;
    if (cudaGraphInstantiate(&ex, g, 0) != cudaSuccess) {
        cudaGraphDestroy(g);
        return STEGO_E_CUDA;
    }
    stego_graph *h = new stego_graph;
    h->graph = g;
    h->exec = ex;
    *out = h;
    return STEGO_OK;
}

int stego_graph_launch(stego_graph *g, void *stream)
{
    if (!g)
        return STEGO_E_INVAL;
    return cudaGraphLaunch(g->exec, (cudaStream_t)stream) == cudaSuccess ? STEGO_OK : STEGO_E_CUDA;
}

int stego_graph_destroy(stego_graph *g)
{
    if (!g)
        return STEGO_OK;
    cudaGraphExecDestroy(g->exec);
    cudaGraphDestroy(g->graph);
    delete g;
    return STEGO_OK;
}

} // extern "C"

// ---------------------------------------------------------------------------
// Batched embed for callers that cannot allocate device memory
// ---------------------------------------------------------------------------
// Some callers cannot call cudaMalloc at all: a host program with no device
// allocator of its own, or one that may not add cudaMalloc's implicit device
// synchronisation to its per-request path.  They still own descriptors,
// covers, messages and results; only the batched call's scratch (tile
// counter, tile offsets, per-cover sizes) moves into this file-scope array,
// sized for STEGO_NOALLOC_MAX_DESCS covers.  Every GPU that loads the library
// holds it until the process exits.

namespace {

constexpr uint32_t kNoAllocMaxDescs = STEGO_NOALLOC_MAX_DESCS;
constexpr uint64_t kNoAllocBytes =
    stego::info_off(kNoAllocMaxDescs) + sizeof(stego::DescInfo) * (uint64_t)kNoAllocMaxDescs;
constexpr int kNoAllocDevices = 64;

std::mutex g_noalloc_mu;
void *g_noalloc_ptr[kNoAllocDevices];              // device address of the array, per device
unsigned long long g_noalloc_ctx[kNoAllocDevices]; // the context that address belongs to

} // namespace

// In host code this name is only a host-side stand-in for the device array:
// the kernels get the address that cudaGetSymbolAddress returns.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

namespace {

// Device address of the scratch array on the current device, looked up once
// per device with that device current, and again after the device was reset
// (its context changed: the module, and with it the array, was loaded anew).
int noalloc_scratch(void **out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess)
        return STEGO_E_CUDA;
    if (dev < 0 || dev >= kNoAllocDevices)
        return STEGO_E_INVAL;
    const unsigned long long ctx = stego::context_id();
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev] || !ctx || g_noalloc_ctx[dev] != ctx) {
        void *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p)
            return STEGO_E_CUDA;
        g_noalloc_ptr[dev] = p;
        g_noalloc_ctx[dev] = ctx;
    }
    *out = g_noalloc_ptr[dev];
    return STEGO_OK;
}

} // namespace

extern "C" int stego_embed_batched_noalloc(const stego_desc *d_descs, uint32_t n,
                                           stego_result *d_results, uint32_t flags,
                                           const stego_tune *tune, void *stream)
{
    stego::Trace trace_("stego_embed_batched_noalloc");
    // argument errors first, as stego_embed_batched reports them
    if (flags & ~(uint32_t)STEGO_FUSE_STATS)
        return STEGO_E_INVAL;
    if (tune && !stego::tune_ok(tune))
        return STEGO_E_INVAL;
    if (n > kNoAllocMaxDescs)
        return STEGO_E_NOMEM;
    if (n == 0)
        return STEGO_OK;
    void *ws = nullptr;
    const int st = noalloc_scratch(&ws);
    if (st != STEGO_OK)
        return st;
    // the preparation launch rewrites every scratch word the persistent
    // kernels read, so the previous call's contents need no clearing
    return stego::batched<true>(d_descs, n, d_results, flags, tune, ws, kNoAllocBytes, stream);
}

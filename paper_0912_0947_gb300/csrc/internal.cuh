// internal.cuh -- declarations shared by the CUDA translation units of
// libstego.so (not part of the public ABI; see include/stego.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include "stego.h"

namespace stego {

// A named range on the calling host thread for profilers and tracers that
// attach through NVTX (nothing but a pointer test when none is attached):
// every entry point, batch and pipeline chunk opens one.
struct Trace {
    explicit Trace(const char *name) { nvtxRangePushA(name); }
    ~Trace() { nvtxRangePop(); }
    Trace(const Trace &) = delete;
    Trace &operator=(const Trace &) = delete;
};

// ---------------------------------------------------------------------------
// Launch shapes
// ---------------------------------------------------------------------------

struct Shape {
    int threads;         // threads per CTA
    int vec;             // 16-byte vectors per thread per loop iteration
    int ctas_per_sm;     // 0 = as many as occupancy allows
    uint32_t tile_bytes; // batched: cover bytes per tile; single-cover STREAM1:
                         // 0 = register kernels, else ring bytes per CTA of
                         // the shared-memory staged kernels
};

// The shape installed for `op`, with the fields of `override_` (if non-null
// and non-zero) taking precedence.
Shape shape_for(int op, const stego_tune *override_);

// Field ranges of a caller-supplied launch shape are valid.
bool tune_ok(const stego_tune *t);

// Number of SMs of the current device (cached per device).
int sm_count();

// Identity of the current CUDA context (process-unique, never reused), or 0
// when it cannot be read.  Caches of device addresses (module globals) are
// keyed on it: a device reset gives the device a new context, in which the
// library's module is loaded again.
unsigned long long context_id();

// Persistent grid: min(ceil(units / units_per_cta), SMs * resident CTAs).
// `kernel` is the __global__ function (for the occupancy query).
int persistent_grid(const void *kernel, int threads, size_t smem, int ctas_per_sm,
                    uint64_t units, uint64_t units_per_cta);

// Grid of a kernel that does units_per_cta units per CTA, however many CTAs these
// make (fewer than 2^31), and adds nothing up: dealt out in order by the hardware,
// the CTAs in flight work on one moving window of memory (a plain copy of 201 MB
// back to back: 61 us, 66-68 us as a persistent grid whose CTAs drift apart).  Only
// where the work is known when the kernel is launched: CTAs that find nothing to do
// cost some 2.5 us for each wave of them.
int one_pass_grid(uint64_t units, uint64_t units_per_cta);

struct StatSlot;

// Programmatic dependent launch: the kernel may be launched while the kernel
// before it in the stream is still finishing (its CTAs then wait on the SMs
// instead of behind the launch).  Only for kernels that call
// grid_dependency_wait() before their first global memory access.
// cluster > 1: CTAs per thread block cluster (the grid a multiple of it).
cudaError_t launch_dependent(const void *kernel, dim3 grid, dim3 block, void **args,
                             size_t smem, cudaStream_t s, uint32_t cluster = 1);

// Launch of a kernel that adds to the two totals at `totals` (nullptr: a kernel
// that does not, launched as a dependent): through the stream's slot, as a dependent
// too; without one the totals are zeroed first, and the kernel is then an ordinary
// launch.  (A dependent behind a memset was in a queue of 300 streams that stopped,
// each a 256 MB copy, a memset and a dependent of 256 CTAs.  It was not found to be
// the cause; CTAs that wait on the SMs for something other than a kernel
// are the one thing that set that queue apart, and they are not needed.)
cudaError_t launch_counting(const void *kernel, dim3 grid, dim3 block, void **args, size_t smem,
                            cudaStream_t s, void *totals, const StatSlot *slot);

// Returns once the grid before this one in the stream has completed and its
// memory operations are visible (at once when there is none, or when the
// launch was an ordinary one).
__device__ __forceinline__ void grid_dependency_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Lets the next kernel in the stream that was launched with
// launch_dependent start launching (it still waits for this grid's end in
// its own grid_dependency_wait()).
__device__ __forceinline__ void allow_dependents()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Fused statistics without a zeroing copy
// ---------------------------------------------------------------------------

// Accumulator of one launch's changed-byte count and squared error and its tile
// counter, one per stream (a static device array, zero at load).  Every CTA
// adds its partial totals and then takes a ticket; the CTA with the last
// ticket moves the totals into the result and clears the slot for the stream's
// next launch.
struct StatSlot {
    unsigned long long changed;
    unsigned long long sse;
    unsigned int arrived;
    unsigned int next; // tiles claimed beyond each CTA's first (for_tiles)
    unsigned long long pad;
};

// What a slot is taken for.  The uses have slots of their own, so that streams
// that only compare, or embed without statistics, leave the statistics theirs.
enum class SlotUse {
    kStats, // an embed's fused statistics (and its tile counter)
    kOther, // a comparison's totals; the tile counter of an embed without statistics
    kCount
};

// The slot of stream s on the current device, or nullptr: then totals are
// zeroed before the launch and the CTAs add into them, and tiles are not claimed.
// Taken only by calls that use it (it costs them some queries of the stream).
// Slots are keyed by the stream's ID (cudaStreamGetId), which the runtime
// never reuses, so a stream created after another was destroyed never
// shares the old stream's slot (whose last launch may still be running).
// nullptr for streams being captured into a graph (a replay may run beside
// direct calls on the same stream), for the per-thread default stream
// (one handle, several streams) and once every slot of the use is taken (256
// streams per device; slots are never handed back, the later streams take the
// zeroing path).
StatSlot *stats_slot(cudaStream_t s, SlotUse use);

// ---------------------------------------------------------------------------
// Launchers (all stream-ordered, no synchronisation).  They return the CUDA
// error of the launch.  `res` (nullable) receives msg_bytes = res_msg_bytes
// and status STEGO_OK from block 0 of the launch; with `stats`, res->changed
// and res->sse accumulate the changed-byte count and squared error (see
// launch_counting).  `slot` is the stream's slot for statistics, or nullptr.
// ---------------------------------------------------------------------------

// STREAM1 embed.  n_bytes: bytes written (C out of place, T in place).
// t_bytes: carrying bytes T = 8 * slen, slen = stream length in bytes
// (message plus 4 header bytes when `header`).  nbits: the header value.
cudaError_t s1_embed(const uint8_t *cover, uint8_t *stego, uint64_t n_bytes, uint64_t t_bytes,
                     const uint8_t *msg, uint64_t slen, bool header, uint32_t nbits, bool stats,
                     stego_result *res, uint64_t res_msg_bytes, const Shape &sh, cudaStream_t s,
                     StatSlot *slot = nullptr);

// STREAM1 extract.  With `header`, the length comes from the stego and all
// fields of `res` (required) are written by block 0; otherwise raw_len bytes
// are extracted and `res` is optional.
cudaError_t s1_extract(const uint8_t *st, uint64_t C, uint8_t *msg, uint64_t cap,
                       uint64_t raw_len, bool header, stego_result *res, const Shape &sh,
                       cudaStream_t s);

// PAPER2 (Sections VI/VII), N > 0.  The embed writes only the 4N plane bytes
// it carries: out of place the caller has copied the cover into stego first.
cudaError_t p2_embed(const uint8_t *cover, uint8_t *stego, const stego_geom &g,
                     const uint8_t *msg, uint64_t N, bool stats, stego_result *res,
                     const Shape &sh, cudaStream_t s, StatSlot *slot = nullptr);
cudaError_t p2_extract(const uint8_t *st, const stego_geom &g, uint8_t *msg, uint64_t N,
                       stego_result *res, const Shape &sh, cudaStream_t s);

// PAPER2 out of place in one pass (copy and embed fused), for 1, 3 or 4
// channels: any row length and any addresses.  N may be 0 (a copy).  Returns
// false with nothing launched when the layout is not one of these (another
// channel count, an image of less than a few vectors); else *err is the
// launch's error.
bool p2_embed_fused(const uint8_t *cover, uint8_t *stego, const stego_geom &g,
                    const uint8_t *msg, uint64_t N, bool stats, stego_result *res,
                    cudaStream_t s, StatSlot *slot, cudaError_t *err);

// STREAM1 with k = 1..4 bits per carrying byte, over all bytes or one plane
// (k >= 2 or plane_only; k = 1 over all bytes is s1_embed).
cudaError_t sk_embed(const uint8_t *cover, uint8_t *stego, uint64_t C, uint32_t k, bool plane_only,
                     const stego_geom *g, const uint8_t *msg, uint64_t m, bool header,
                     bool stats, stego_result *res, const Shape &sh, cudaStream_t s,
                     StatSlot *slot = nullptr);
cudaError_t sk_extract(const uint8_t *st, uint64_t C, uint32_t k, bool plane_only,
                       const stego_geom *g, uint8_t *msg, uint64_t cap, uint64_t raw_len,
                       bool header, stego_result *res, const Shape &sh, cudaStream_t s);

// STREAM1 extraction with the message packed by warp ballots (one stego
// byte per lane; ballot.cu); same arguments and results as s1_extract.
cudaError_t s1_extract_ballot(const uint8_t *st, uint64_t C, uint8_t *msg, uint64_t cap,
                              uint64_t raw_len, bool header, stego_result *res, const Shape &sh,
                              cudaStream_t s);

// STREAM1 kernels staged through shared memory with bulk asynchronous
// copies (bulk.cu); same arguments and results as s1_embed / s1_extract.
// Usable with 16-byte aligned buffers when bulk_stages(sh) >= 2: a shape
// with tile_bytes = ring bytes per CTA, tiles of threads * 16 * vec bytes.
uint32_t bulk_stages(const Shape &sh);
cudaError_t s1_embed_bulk(const uint8_t *cover, uint8_t *stego, uint64_t n_bytes,
                          uint64_t t_bytes, const uint8_t *msg, uint64_t slen, bool header,
                          uint32_t nbits, bool stats, stego_result *res, uint64_t res_msg_bytes,
                          const Shape &sh, cudaStream_t s, StatSlot *slot = nullptr);
cudaError_t s1_extract_bulk(const uint8_t *st, uint64_t C, uint8_t *msg, uint64_t cap,
                            uint64_t raw_len, bool header, stego_result *res, const Shape &sh,
                            cudaStream_t s);

// Changed-byte count and SSE of two arrays into out2[0..1].
cudaError_t changed_bytes(const uint8_t *a, const uint8_t *b, uint64_t n,
                          unsigned long long *out2, const Shape &sh, cudaStream_t s,
                          StatSlot *slot);

// One thread writes a whole result (calls that launch no other kernel).
cudaError_t write_result(stego_result *res, uint64_t msg_bytes, int status, cudaStream_t s);

// ---------------------------------------------------------------------------
// Device helpers
// ---------------------------------------------------------------------------

// Adds (a, b) of every thread of the block into out[0], out[1] with one pair
// of 64-bit atomics per block.  All threads of the block must call it.
__device__ __forceinline__ void block_add2(unsigned long long a, unsigned long long b,
                                           unsigned long long *out)
{
    __shared__ unsigned long long sa[32], sb[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xFFFFFFFFu, a, o);
        b += __shfl_down_sync(0xFFFFFFFFu, b, o);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) {
        sa[w] = a;
        sb[w] = b;
    }
    __syncthreads();
    if (w == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        a = lane < nw ? sa[lane] : 0ull;
        b = lane < nw ? sb[lane] : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xFFFFFFFFu, a, o);
            b += __shfl_down_sync(0xFFFFFFFFu, b, o);
        }
        if (lane == 0) {
            if (a)
                atomicAdd(out, a);
            if (b)
                atomicAdd(out + 1, b);
        }
    }
}

// The statistics of a single-cover launch: the block's totals go into
// res->changed/sse (zeroed by the caller) without a slot, or into the slot,
// whose last arriving CTA writes res->changed/sse.  All threads of every
// CTA of the grid must call it once.
__device__ __forceinline__ void block_stats(unsigned long long a, unsigned long long b,
                                            stego_result *res, StatSlot *slot)
{
    if (!slot) {
        block_add2(a, b, reinterpret_cast<unsigned long long *>(&res->changed));
        return;
    }
    __shared__ unsigned long long sa[32], sb[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xFFFFFFFFu, a, o);
        b += __shfl_down_sync(0xFFFFFFFFu, b, o);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) {
        sa[w] = a;
        sb[w] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        a = 0;
        b = 0;
        for (int i = 0; i < nw; ++i) {
            a += sa[i];
            b += sb[i];
        }
        if (a)
            atomicAdd(&slot->changed, a);
        if (b)
            atomicAdd(&slot->sse, b);
        __threadfence(); // the adds are visible before the ticket
        if (atomicAdd(&slot->arrived, 1u) == gridDim.x - 1) {
            __threadfence();
            res->changed = atomicExch(&slot->changed, 0ull);
            res->sse = atomicExch(&slot->sse, 0ull);
            atomicExch(&slot->next, 0u);
            atomicExch(&slot->arrived, 0u);
        }
    }
}

// Whether tiles are claimed: with a slot, and more than four for each CTA (with
// fewer the CTAs have no time to drift, and the barrier per tile costs more:
// 25 MB at odd addresses 12.0 us, 13.3 claimed).
__host__ __device__ __forceinline__ bool enough_tiles(uint64_t ntiles, uint32_t ctas)
{
    return ntiles > 4ull * ctas;
}
__device__ __forceinline__ bool tiles_claimed(const StatSlot *slot, uint32_t ntiles)
{
    return slot && enough_tiles(ntiles, gridDim.x);
}

// Calls body(tile) for this CTA's tiles of ntiles, all its threads together:
// the tile of its own index, then the next one that no CTA has taken yet
// (tiles_claimed), else every gridDim.x-th.  Taken in order the tiles in flight stay
// one moving window of memory: dealt by the grid's stride the CTAs drift apart
// (a plain copy of 201 MB back to back: 66-68 us by stride, 61 us as one CTA per
// tile; but a CTA per tile adds its statistics for each, three atomics on one
// address, 70 -> 78 us for the one-bit embed).  The next claim is in flight
// while a tile is worked on.  After it every CTA calls block_stats or
// tiles_done once.  It pays where a kernel does little but move data: the k-bit
// and paper-layout units and the comparison of two arrays measured slower
// (8192x8192x3: k = 2 77 -> 80 us, one channel of the paper's layout 31 -> 34,
// comparison 58 -> 63).
template <typename Body>
__device__ __forceinline__ void for_tiles(StatSlot *slot, uint32_t ntiles, Body &&body)
{
    __shared__ uint32_t s_next[2];
    const bool claims = tiles_claimed(slot, ntiles);
    uint32_t i = 0;
    for (uint32_t tile = blockIdx.x; tile < ntiles;) {
        uint32_t next = tile + gridDim.x;
        if (claims && threadIdx.x == 0)
            next = gridDim.x + atomicAdd(&slot->next, 1u);
        body(tile);
        if (claims) {
            if (threadIdx.x == 0)
                s_next[i] = next;
            __syncthreads(); // (two words: the next write is two barriers from this read)
            next = s_next[i];
            i ^= 1u;
        }
        tile = next;
    }
}

// Clears the tile counter for the stream's next launch (kernels that do not
// call block_stats).
__device__ __forceinline__ void tiles_done(StatSlot *slot, uint32_t ntiles)
{
    if (tiles_claimed(slot, ntiles) && threadIdx.x == 0) {
        __threadfence(); // this CTA's claims are done before its ticket
        if (atomicAdd(&slot->arrived, 1u) == gridDim.x - 1) {
            atomicExch(&slot->next, 0u);
            atomicExch(&slot->arrived, 0u);
        }
    }
}

// Changed bytes and squared error of a unit's 16 carrying bytes (c before,
// o after, d = o ^ c, differences in the low K bits only), summed in 32 bits
// per unit.  A byte changed when any of its low K bits did (the packing and
// the per-field test are below).  With K = 1 every change is +-1, so the
// squared error equals the count.
template <int K>
__device__ __forceinline__ void unit_stats(const uint32_t (&o)[4], const uint32_t (&c)[4],
                                           const uint32_t (&d)[4], uint32_t kmul,
                                           unsigned long long &changed,
                                           unsigned long long &sse)
{
    constexpr uint32_t BM = ((1u << K) - 1u) * 0x01010101u;
    uint32_t n, s = 0;
    static_assert(K >= 1 && K <= 4, "one to four bits per byte");
    if constexpr (K <= 2) {
        // the four words' K-bit changes in disjoint bit ranges of each byte
        // (word i at bits K*i), joined by multiply-adds, then one fold
        // Horner in kmul = 1 << K: multiply-adds (FMA pipe), not shifts on
        // the busy ALU pipe; kmul comes from the launch arguments so the
        // compiler keeps the multiplies
        const uint32_t acc0 = ((d[3] * kmul + d[2]) * kmul + d[1]) * kmul + d[0];
        uint32_t acc = acc0;
        if (K == 2)
            acc = (acc | (acc >> 1)) & 0x55555555u;
        n = __popc(acc);
    } else {
        // k = 3, 4: two words per byte (word 2j+1 at bit K), then a field is
        // nonzero when its top bit is set or its low K-1 bits plus all ones
        // carry into the top bit (no carry leaves a field)
        constexpr uint32_t LOW = K == 4 ? 0x77777777u : 0x1B1B1B1Bu;
        constexpr uint32_t TOP = K == 4 ? 0x88888888u : 0x24242424u;
        const uint32_t a01 = d[1] * kmul + d[0], a23 = d[3] * kmul + d[2];
        n = __popc((a01 | ((a01 & LOW) + LOW)) & TOP) + __popc((a23 | ((a23 & LOW) + LOW)) & TOP);
    }
    if (K > 1) {
        uint32_t ab = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) { // sum of (a - b)^2 = a.a + b.b - 2 a.b over the fields
            const uint32_t fa = o[i] & BM, fb = c[i] & BM;
            s = __dp4a(fa, fa, s);
            s = __dp4a(fb, fb, s);
            ab = __dp4a(fa, fb, ab);
        }
        s -= 2u * ab;
    }
    changed += n;
    sse += K > 1 ? s : n;
}

// Warp staging of pixel units (16 pixels of CH channels = CH 16-byte
// vectors): a warp's 32 consecutive units are loaded and stored in memory
// order and exchanged through shared memory, SV = unit_stage_slots<CH>()
// slots per warp.  Vector v of the warp's units sits in slot
// unit_stage_slot<CH>(v); CH = 4 pads one slot per 8 so that both the
// memory-order (v = 32j + lane) and the unit-order (v = CH*lane + q)
// accesses are free of bank conflicts (CH = 3 needs no padding).
template <int CH>
__host__ __device__ constexpr uint32_t unit_stage_slots()
{
    return 32 * CH + (CH == 4 ? 16 : 0);
}

template <int CH>
__device__ __forceinline__ uint32_t unit_stage_slot(uint32_t v)
{
    return CH == 4 ? v + (v >> 3) : v;
}

} // namespace stego


// S1 — mask compaction: kept[j] = position of the j-th non-zero mask byte, ascending.
//
// Appendix A, Algorithm 2 (first function) walks the output positions in raster order and
// appends an entry for every position whose mask is 1; the running index of that loop is an
// exclusive prefix sum of the mask.  Here the prefix sum has two levels: inside a 16384-row
// tile (4 x 16 mask bytes per thread, popcount, a shuffle scan inside each warp and across the
// warp totals) and across runs of tiles (one run per resident block: a counting pass, then a
// writing pass in which every block sums the counts in front of its run).  Small masks take one
// pass in which every block counts all mask bytes in front of its own 4096.
#include "asx_internal.h"
#include "ptx_sm100.cuh"

namespace asx {

namespace {

struct ScratchHeader {       // first 8 bytes of the scratch; the tile counts follow
    unsigned int reserved;   // kept zero
    int error;               // device status word of the compaction (kept zero: nothing here can time out)
};

// The sixteen flags of one 16-byte load, one bit per mask byte, in the order the arithmetic gives them
// cheapest: byte b of word k (row 4 k + b of the sixteen) lands on bit 8 b + k.
__device__ __forceinline__ constexpr int flag_bit(int j) { return 8 * (j & 3) + (j >> 2); }

__device__ __forceinline__ unsigned nonzero_flags16(const uint4& v)
{
    const unsigned w[4] = {v.x, v.y, v.z, v.w};
    unsigned u = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned t = ((w[k] & 0x7f7f7f7fu) + 0x7f7f7f7fu) | w[k];     // bit 7 of each byte: byte != 0
        u |= (t >> (7 - k)) & (0x01010101u << k);
    }
    return u;
}

// A block takes COMPACT_SUB consecutive 4096-row sub-tiles and loads all their mask bytes before
// anything else: four 16-byte loads in flight per thread instead of one.
// Where that would leave SMs without a block (up to 4.8 million rows) a block takes one sub-tile.
constexpr int COMPACT_SUB = 4;
constexpr int COMPACT_RESIDENT = 8;      // blocks per SM of the two passes over a large mask
constexpr int64_t COMPACT_PREFIX_MAX_ROWS = 192 * 1024;

// ---- Large masks: two passes over a grid of resident blocks, no block ever waits for another.  Block g
// owns a run of consecutive tiles of SUB sub-tiles.  Pass 1 counts the kept rows of every run; in pass 2 a block
// adds up the counts of the runs in front of its own (a few loads per thread, all L2 hits), then writes
// its tiles' indices one tile after another, carrying the offset along.  The mask is read twice, i.e.
// `rows` more bytes than a single-pass chained scan (tiles that publish their totals and look back over
// their predecessors' status words) would move; that form was built first and measured slower (0.150-0.152
// ms on 2^27 rows), and it needs a ticket, cleared status words and bounded spin-waits, which this one
// does not.
template <int SUB>
__device__ __forceinline__ void load_tile_flags(const uint8_t* __restrict__ mask, long long rows, long long tile_first,
                                                int tid, unsigned (&flags)[SUB])
{
    const bool aligned = (reinterpret_cast<uintptr_t>(mask) & 15) == 0;
    uint4 raw[SUB];
    bool fast[SUB];
#pragma unroll
    for (int sub = 0; sub < SUB; ++sub) {
        const long long first = tile_first + (long long)sub * COMPACT_TILE + (long long)tid * COMPACT_PER_THREAD;
        fast[sub] = aligned && first + COMPACT_PER_THREAD <= rows;
        raw[sub] = make_uint4(0, 0, 0, 0);
        if (fast[sub]) raw[sub] = __ldcg(reinterpret_cast<const uint4*>(mask + first));     // past L1: a kernel may have written the mask
    }
#pragma unroll
    for (int sub = 0; sub < SUB; ++sub) {
        const long long first = tile_first + (long long)sub * COMPACT_TILE + (long long)tid * COMPACT_PER_THREAD;
        unsigned f = 0;
        if (fast[sub]) {
            f = nonzero_flags16(raw[sub]);
        } else {
            for (int j = 0; j < COMPACT_PER_THREAD; ++j)
                if (first + j < rows && __ldcg(mask + first + j) != 0) f |= 1u << flag_bit(j);
        }
        flags[sub] = f;
    }
}

__device__ __forceinline__ void run_of_block(int tiles, int& t0, int& t1)
{
    t0 = (int)((long long)tiles * blockIdx.x / gridDim.x);
    t1 = (int)((long long)tiles * (blockIdx.x + 1) / gridDim.x);
}

// Sum of v over the block, returned to every thread (two barriers).
__device__ __forceinline__ int block_sum(int v, int* s_warp, int* s_total)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    if (lane == 0) s_warp[warp] = v;
    __syncthreads();
    if (tid == 0) {
        int t = 0;
#pragma unroll
        for (int i = 0; i < COMPACT_THREADS / 32; ++i) t += s_warp[i];
        *s_total = t;
    }
    __syncthreads();
    return *s_total;
}

template <int SUB>
__global__ void __launch_bounds__(COMPACT_THREADS, COMPACT_RESIDENT)
compact_count_kernel(const uint8_t* __restrict__ mask, long long rows, int tiles, unsigned* __restrict__ run_count)
{
    __shared__ int s_warp[COMPACT_THREADS / 32];
    __shared__ int s_total;
    const int tid = threadIdx.x;
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();          // the scratch may still be read by an earlier call's kernels
    int t0, t1;
    run_of_block(tiles, t0, t1);
    int v = 0;
    for (int t = t0; t < t1; ++t) {
        unsigned flags[SUB];
        load_tile_flags(mask, rows, (long long)t * (SUB * COMPACT_TILE), tid, flags);
#pragma unroll
        for (int sub = 0; sub < SUB; ++sub) v += __popc(flags[sub]);
    }
    const int total = block_sum(v, s_warp, &s_total);
    if (tid == 0) run_count[blockIdx.x] = (unsigned)total;
}

// Pass 1 of asx_set_mask with a device mask: the same counts, and the mask's bytes into the layer's own buffer on the way.
// (A device-to-device copy in front of pass 1 cost 3.4 us and, as no kernel, kept both its neighbours from overlapping.)
template <int SUB>
__global__ void __launch_bounds__(COMPACT_THREADS, COMPACT_RESIDENT)
compact_copy_count_kernel(const uint8_t* __restrict__ mask, long long rows, int tiles, uint8_t* __restrict__ copy, unsigned* __restrict__ run_count)
{
    __shared__ int s_warp[COMPACT_THREADS / 32];
    __shared__ int s_total;
    const int tid = threadIdx.x;
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();          // the mask may come from the kernel before; the layer's buffer may still be read
    int t0, t1;
    run_of_block(tiles, t0, t1);
    const bool aligned = (reinterpret_cast<uintptr_t>(mask) & 15) == 0;        // the copy is an allocation of its own
    const long long end = (long long)t1 * (SUB * COMPACT_TILE) < rows ? (long long)t1 * (SUB * COMPACT_TILE) : rows;
    int v = 0;
#pragma unroll 4
    for (long long first = (long long)t0 * (SUB * COMPACT_TILE) + tid * COMPACT_PER_THREAD; first < end; first += COMPACT_TILE) {
        if (aligned && first + COMPACT_PER_THREAD <= rows) {
            const uint4 m = __ldcg(reinterpret_cast<const uint4*>(mask + first));
            *reinterpret_cast<uint4*>(copy + first) = m;
            v += __popc(nonzero_flags16(m));
        } else {
            for (int j = 0; j < COMPACT_PER_THREAD && first + j < rows; ++j) {
                const uint8_t m = __ldcg(mask + first + j);
                copy[first + j] = m;
                v += m != 0;
            }
        }
    }
    const int total = block_sum(v, s_warp, &s_total);
    if (tid == 0) run_count[blockIdx.x] = (unsigned)total;
}

// Pass 2: the indices of a 4096-row sub-tile are put in order in shared memory and copied to the list
// with full-width stores (direct stores of each 32-row ballot word's indices, without the staging,
// write half-filled lines and were 12 % slower; 16-byte stores from the unaligned staging buffer 3 %; a
// staging index swizzled against bank conflicts 18 %).  On 2^27 rows, half of them kept, the shared-memory pipe is busy 75 % of
// the time (two thirds of it the staging stores, more than half of those bank conflicts), the issue slots 67 %, DRAM 46 %.
// EARLY_MASK: no kernel that may still be running wrote the mask (a layer's own copy of its mask, unless it has just been taken
// from the device), so the first tile's mask bytes may be loaded and scanned before the dependency wait, while the pass before
// still runs.  A caller's mask buffer may have been written by the kernel just before this call (a
// data-dependent mask), which, launched as a programmatic predecessor, can still be storing it: then the
// load waits like everything else.
template <int SUB, bool EARLY_MASK>
__global__ void __launch_bounds__(COMPACT_THREADS, COMPACT_RESIDENT)
compact_write_kernel(const uint8_t* __restrict__ mask, long long rows, int tiles, int32_t* __restrict__ kept,
                     const unsigned* __restrict__ run_count, int32_t* __restrict__ count, ScratchHeader* hdr)
{
    __shared__ int32_t s_idx[COMPACT_TILE];
    __shared__ int s_warp_total[SUB][COMPACT_THREADS / 32];
    __shared__ int s_total;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    ptx::grid_launch_dependents();
    int t0, t1;
    run_of_block(tiles, t0, t1);
    unsigned flags[SUB];
    if (!EARLY_MASK) ptx::grid_dependency_wait();
    if (t0 < t1) load_tile_flags(mask, rows, (long long)t0 * (SUB * COMPACT_TILE), tid, flags);
    if (EARLY_MASK) ptx::grid_dependency_wait();          // the counts come from the pass before; the list may still be read
    // Offset of this block's run: the counts of all runs in front of it.  Read past L1: this block was
    // launched while the pass before was running, L1 is not invalidated in between, and the SM may hold
    // a stale line of the scratch.
    int before = 0;
    for (int i = tid; i < (int)blockIdx.x; i += COMPACT_THREADS) before += (int)__ldcg(run_count + i);
    int exclusive = block_sum(before, s_warp_total[0], &s_total);
    for (int t = t0; t < t1; ++t) {
        const long long tile_first = (long long)t * (SUB * COMPACT_TILE);
        if (t != t0) load_tile_flags(mask, rows, tile_first, tid, flags);
        int mine[SUB], incl[SUB];
#pragma unroll
        for (int sub = 0; sub < SUB; ++sub) {
            mine[sub] = __popc(flags[sub]);
            int v = mine[sub];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, d);
                if (lane >= d) v += u;
            }
            incl[sub] = v;
            if (lane == 31) s_warp_total[sub][warp] = v;
        }
        __syncthreads();
#pragma unroll
        for (int sub = 0; sub < SUB; ++sub) {
            // lanes 0..7 hold the eight warp totals; a three-step scan gives every warp its prefix and the tile total
            const int wt = lane < COMPACT_THREADS / 32 ? s_warp_total[sub][lane] : 0;
            int winc = wt;
#pragma unroll
            for (int d = 1; d < COMPACT_THREADS / 32; d <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, winc, d);
                if (lane >= d) winc += u;
            }
            const int wp = __shfl_sync(0xffffffffu, winc - wt, warp);
            const int tot = __shfl_sync(0xffffffffu, winc, COMPACT_THREADS / 32 - 1);
            const long long first = tile_first + (long long)sub * COMPACT_TILE + (long long)tid * COMPACT_PER_THREAD;
            const int at = wp + incl[sub] - mine[sub];
            const unsigned f = flags[sub];
            if (f) {                                               // sixteen predicated stores, no loop over set bits
                int pos = at;
                const int32_t v0 = (int32_t)first;
#pragma unroll
                for (int j = 0; j < COMPACT_PER_THREAD; ++j)
                    if ((f >> flag_bit(j)) & 1u) { s_idx[pos] = v0 + j; ++pos; }
            }
            __syncthreads();
            {
                int32_t* dst = kept + exclusive;
                int i = tid;
                for (; i + 3 * COMPACT_THREADS < tot; i += 4 * COMPACT_THREADS) {      // four loads ahead of four stores
                    const int32_t a0 = s_idx[i], a1 = s_idx[i + COMPACT_THREADS], a2 = s_idx[i + 2 * COMPACT_THREADS],
                                  a3 = s_idx[i + 3 * COMPACT_THREADS];
                    dst[i] = a0;
                    dst[i + COMPACT_THREADS] = a1;
                    dst[i + 2 * COMPACT_THREADS] = a2;
                    dst[i + 3 * COMPACT_THREADS] = a3;
                }
                for (; i < tot; i += COMPACT_THREADS) dst[i] = s_idx[i];
            }
            exclusive += tot;
            __syncthreads();                                       // s_idx and, after the last sub-tile, the warp totals are reused
        }
    }
    if (blockIdx.x == gridDim.x - 1 && tid == 0) {
        *count = (int32_t)exclusive;
        hdr->reserved = 0;                   // a status query must find a clean word
        hdr->error = 0;
    }
}

// Small masks: one pass, one 4096-row sub-tile per block; the number of kept rows in front of it every block counts
// itself, from the mask (up to 192 KB out of L2, loads in flight together, beside its own tile's scan), so no block needs
// another one's result and there is one launch instead of two.
__global__ void __launch_bounds__(COMPACT_THREADS)
compact_prefix_kernel(const uint8_t* __restrict__ mask, int rows, int32_t* __restrict__ kept, int32_t* __restrict__ count,
                      ScratchHeader* hdr, uint8_t* __restrict__ copy, int early_mask)
{
    __shared__ int32_t s_idx[COMPACT_TILE];
    __shared__ int s_own[COMPACT_THREADS / 32], s_before[COMPACT_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    ptx::grid_launch_dependents();
    if (!early_mask) ptx::grid_dependency_wait();         // see compact_write_kernel
    const bool aligned = (reinterpret_cast<uintptr_t>(mask) & 15) == 0;
    const int tile_first = blockIdx.x * COMPACT_TILE, first = tile_first + tid * COMPACT_PER_THREAD;
    unsigned flags = 0;
    if (aligned && first + COMPACT_PER_THREAD <= rows) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4*>(mask + first));      // past L1: a kernel may have written the mask
        if (copy != nullptr) *reinterpret_cast<uint4*>(copy + first) = v;
        flags = nonzero_flags16(v);
    } else {
        for (int j = 0; j < COMPACT_PER_THREAD && first + j < rows; ++j) {
            const uint8_t m = __ldcg(mask + first + j);
            if (copy != nullptr) copy[first + j] = m;
            if (m != 0) flags |= 1u << flag_bit(j);
        }
    }
    int before = 0;
    if (aligned) {
#pragma unroll 8
        for (int i = tid * COMPACT_PER_THREAD; i < tile_first; i += COMPACT_TILE)
            before += __popc(nonzero_flags16(__ldcg(reinterpret_cast<const uint4*>(mask + i))));
    } else {
#pragma unroll 8
        for (int i = tid; i < tile_first; i += COMPACT_THREADS) before += __ldcg(mask + i) != 0;
    }
    const int mine = __popc(flags);
    int incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 31) { s_own[warp] = incl; s_before[warp] = before; }
    __syncthreads();
    int at = incl - mine, tot = 0, exclusive = 0;
#pragma unroll
    for (int i = 0; i < COMPACT_THREADS / 32; ++i) {
        if (i < warp) at += s_own[i];
        tot += s_own[i];
        exclusive += s_before[i];
    }
#pragma unroll
    for (int j = 0; j < COMPACT_PER_THREAD; ++j)
        if ((flags >> flag_bit(j)) & 1u) { s_idx[at] = first + j; ++at; }
    __syncthreads();
    if (early_mask) ptx::grid_dependency_wait();          // the list may still be read
    for (int i = tid; i < tot; i += COMPACT_THREADS) kept[exclusive + i] = s_idx[i];
    if (blockIdx.x == gridDim.x - 1 && tid == 0) {
        *count = exclusive + tot;
        if (hdr != nullptr) { hdr->reserved = 0; hdr->error = 0; }     // a status query must find a clean word
    }
}

}  // namespace

static int resident_sms()               // SM count of the current device (looked up once per device)
{
    static int sms[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    if (sms[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 148;
        sms[dev] = n;
    }
    return sms[dev];
}

static int tiles_for(int64_t rows)      // 4096-row units: sizes the scratch (8 bytes each; the passes use 4 bytes per resident block, at most one block per unit)
{
    int64_t t = (rows + COMPACT_TILE - 1) / COMPACT_TILE;
    return (int)(t < 1 ? 1 : t);
}

int64_t compact_scratch_bytes(int64_t rows)
{
    return (int64_t)sizeof(ScratchHeader) + 8 * (int64_t)tiles_for(rows);
}

template <int SUB>
static cudaError_t launch_two_passes(const uint8_t* mask, int64_t rows, int32_t* kept, int32_t* count, ScratchHeader* hdr, cudaStream_t st,
                                     bool early_mask, uint8_t* copy)
{
    const int tiles = (int)((rows + SUB * COMPACT_TILE - 1) / (SUB * COMPACT_TILE));
    // one resident block per run of tiles: eight blocks per SM, never more blocks than tiles (the scratch has
    // 8 bytes per 4096 rows, i.e. room for two 32-bit counts per sub-tile)
    const int grid = tiles < COMPACT_RESIDENT * resident_sms() ? tiles : COMPACT_RESIDENT * resident_sms();
    unsigned* run_count = reinterpret_cast<unsigned*>(hdr + 1);
    cudaError_t e = copy != nullptr
                        ? launch_pdl(compact_copy_count_kernel<SUB>, dim3(grid), dim3(COMPACT_THREADS), 0, st, mask, (long long)rows, tiles, copy, run_count)
                        : launch_pdl(compact_count_kernel<SUB>, dim3(grid), dim3(COMPACT_THREADS), 0, st, mask, (long long)rows, tiles, run_count);
    if (e == cudaSuccess)
        e = launch_pdl(early_mask ? compact_write_kernel<SUB, true> : compact_write_kernel<SUB, false>, dim3(grid), dim3(COMPACT_THREADS), 0, st,
                       mask, (long long)rows, tiles, kept, static_cast<const unsigned*>(run_count), count, hdr);
    return e;
}

cudaError_t launch_compact(const uint8_t* mask, int64_t rows, int32_t* kept, int32_t* count,
                           void* scratch, cudaStream_t st, bool mask_settled, uint8_t* copy)
{
    auto* hdr = static_cast<ScratchHeader*>(scratch);
    // One pass while counting all bytes in front of the last block costs less than a second launch (about 2 us), and the
    // bytes can be counted sixteen at a time; without that, while they are few.
    const bool aligned = (reinterpret_cast<uintptr_t>(mask) & 15) == 0;
    if (rows <= (aligned ? COMPACT_PREFIX_MAX_ROWS : COMPACT_SMALL_MAX_ROWS))
        return launch_pdl(compact_prefix_kernel, dim3((unsigned)tiles_for(rows)), dim3(COMPACT_THREADS), 0, st, mask,
                          (int)rows, kept, count, hdr, copy, mask_settled ? 1 : 0);
    return rows <= (int64_t)COMPACT_TILE * COMPACT_RESIDENT * resident_sms()
               ? launch_two_passes<1>(mask, rows, kept, count, hdr, st, mask_settled, copy)
               : launch_two_passes<COMPACT_SUB>(mask, rows, kept, count, hdr, st, mask_settled, copy);
}

}  // namespace asx

// ---------------------------------------------------------------------------------------------
// asx_compact_static: the same compaction for callers that must not allocate.
//
// The compaction of a large mask needs a little global scratch (a header and the per-tile counts,
// sized at 8 bytes per 4096 rows).  Every other entry point takes that scratch from the caller or from
// memory the layer allocated.  Some callers can do neither at the moment they need a kept-row
// list: a serving loop that must not call cudaMalloc because it synchronises the whole device and
// stalls every other stream; code running after a framework has claimed all device memory for
// its own pool; a plug-in that only holds the raw buffers its host handed in.  For them the
// scratch lives in the library image itself, in the array below: no allocation call of any
// kind is made, at the price of a fixed upper size and of one array shared between all calls.
namespace {

constexpr long long STATIC_MAX_ROWS = ASX_COMPACT_STATIC_MAX_ROWS;
constexpr size_t STATIC_SCRATCH_BYTES = 8 + 8 * (size_t)(STATIC_MAX_ROWS / asx::COMPACT_TILE);

// Held by every GPU that loads the library until the process exits (about 32 KB).
static __device__ __align__(256) unsigned char g_static_scratch[STATIC_SCRATCH_BYTES];

// In host code `g_static_scratch` is only a handle for the runtime, not an address the GPU
// understands, so the device address is looked up once per device and remembered here.
constexpr int MAX_DEVICES = 64;
void* g_static_scratch_addr[MAX_DEVICES] = {nullptr};

}  // namespace

extern "C" asx_status asx_compact_static(const uint8_t* mask_dev, int64_t rows, int32_t* kept_dev,
                                         int32_t* count_dev, void* cuda_stream)
{
    if (rows < 0 || count_dev == nullptr) return ASX_ERR_INVALID_ARG;
    if (rows > 0 && (mask_dev == nullptr || kept_dev == nullptr)) return ASX_ERR_INVALID_ARG;
    if (rows > STATIC_MAX_ROWS) return ASX_ERR_UNSUPPORTED;          // the built-in scratch is too small
    if ((reinterpret_cast<uintptr_t>(kept_dev) & 3) || (reinterpret_cast<uintptr_t>(count_dev) & 3)) return ASX_ERR_ALIGN;
    if ((size_t)asx::compact_scratch_bytes(rows) > STATIC_SCRATCH_BYTES) return ASX_ERR_UNSUPPORTED;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ASX_ERR_CUDA;
    if (dev < 0 || dev >= MAX_DEVICES) return ASX_ERR_UNSUPPORTED;
    if (g_static_scratch_addr[dev] == nullptr) {
        // first call on this device: resolve the array's device address (not a stream operation)
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || p == nullptr) {
            cudaGetLastError();
            return ASX_ERR_CUDA;
        }
        g_static_scratch_addr[dev] = p;
    }
    // launch_compact overwrites every word of the array it later reads (tile counts, header), in
    // stream order, so whatever the previous call left in the array does not matter.
    return asx::launch_compact(mask_dev, rows, kept_dev, count_dev, g_static_scratch_addr[dev],
                               static_cast<cudaStream_t>(cuda_stream), false, nullptr) == cudaSuccess
               ? ASX_OK
               : ASX_ERR_CUDA;
}

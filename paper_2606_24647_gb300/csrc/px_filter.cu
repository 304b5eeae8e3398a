// px_filter: FilterProject's predicate (Sec. 3.2) as a stream compaction in two
// launches over one wave of blocks each, in tiles of four warps x W words of 32 rows:
//   1. count - the blocks sweep the column together (block b takes tiles b, b + G, ..),
//              store one bit per row (1 where lo <= col < hi) and every tile's passing
//              rows;
//   2. write - each block owns one contiguous run of tiles: it sums the counts of the
//              tiles before it, which gives it its first output slot, reads its bits
//              back and writes the passing rows' numbers in ascending order. Only the
//              bits are read again, and no block waits for another.
// HBM traffic: the column once, 1/8 byte per row of bits written and read, 4 bytes
// per passing row. The write launch overlaps the count's tail (programmatic dependent
// launch). px_filter_noalloc has no room for bits: its write pass reads the column
// again.
// Measured, 60M int32 rows, 30 % kept (312 MB): 154 us when the write pass read the
// column again behind a one-block scan of the tile counts, now 77 us: the count is
// DRAM bound (47 us, 5.2 TB/s; 2.8 TB/s when every block read a contiguous run of its
// own, 12 MB apart), the write issue bound (30 us, 2.8 instructions per cycle). 60M
// int64 rows: 182 -> 123 us; 1M int32 rows 7.4 -> 4.8 us. Prefetching the next tiles
// into L2 (up to 60 MB ahead) evicted lines before their use: int64 166 us.
#include <algorithm>
#include <limits>
#include <mutex>
#include <type_traits>

#include "px_common.cuh"

namespace px {
namespace {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
// 1536 resident threads of 40 registers each: the 32-word kernels of int64 columns spill 72
// bytes (count) and 64 (write), the count of int32 columns 16.
constexpr int kBlocksPerSm = 12;
// Words of 32 rows a warp takes per tile: 32, or 8 while one tile of 8 per block
// holds the rows: a short column then spreads over more warps with fewer serial
// loads each (10,000 int64 rows: 3.6 us, 7.9 us in 32-word tiles).
constexpr int kWide = 32, kNarrow = 8;

// A warp's 1024 rows are staged in shared memory lane by lane while fewer than kDense
// pass, else written word by word (write pass, 60M rows: 30 % kept 30 us staged, 41 us
// by words; 98 % kept 69 us and 48 us).
constexpr uint32_t kDense = 640;
constexpr int kStage = 1024 + 32;      // staged rows of a warp, one word in 33 unused

// Passing values of a T column: x - lo (as unsigned) <= last; `none`: no value passes.
template <typename T>
struct Range {
    T lo;
    std::make_unsigned_t<T> last;
    bool none;
};

// [lo, hi) clamped to T's values.
template <typename T>
Range<T> make_range(int64_t lo, int64_t hi) {
    Range<T> r = {};
    const int64_t tmin = std::numeric_limits<T>::min(), tmax = std::numeric_limits<T>::max();
    const int64_t first = std::max(lo, tmin);
    // the last passing value hi - 1, when there is one
    r.none = hi <= first || first > tmax;
    if (r.none) return r;
    r.lo = static_cast<T>(first);
    r.last = static_cast<std::make_unsigned_t<T>>(static_cast<uint64_t>(std::min(hi - 1, tmax)) -
                                                  static_cast<uint64_t>(first));
    return r;
}

template <typename T>
__device__ __forceinline__ bool passes(T x, const Range<T>& g) {
    using U = std::make_unsigned_t<T>;
    return static_cast<U>(static_cast<U>(x) - static_cast<U>(g.lo)) <= g.last;
}

// This lane's word of the W words from row `base`: bit b of lane l < W is row base +
// 32 l + b. W = 32: 16-byte loads of 16 / 4 / 2 consecutive rows per lane, whose bits
// neighbouring lanes join into words; W = 8: one load and one ballot per word. Rows
// from n on are 0.
template <typename T, int W>
__device__ __forceinline__ uint32_t warp_words(const T* __restrict__ col, int64_t base, int64_t n, const Range<T>& g,
                                               int lane) {
    uint32_t word = 0;
    if (base + 32 * W <= n) {
        if (W == 32) {
            constexpr int kV = 16 / sizeof(T);                 // rows per lane and load
            constexpr int kWordLanes = 32 / kV;                // lanes that make a word
            constexpr int kChunks = 32 / kV;                   // loads per lane
            constexpr int kBatch = kChunks < 8 ? kChunks : 8;  // of them in flight
            const int4* src = reinterpret_cast<const int4*>(col + base) + lane;
#pragma unroll
            for (int h = 0; h < kChunks; h += kBatch) {
                int4 v[kBatch];
#pragma unroll
                for (int k = 0; k < kBatch; ++k) v[k] = src[32 * (h + k)];
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    const T* x = reinterpret_cast<const T*>(&v[k]);
                    uint32_t part = 0;
#pragma unroll
                    for (int j = 0; j < kV; ++j) part |= (passes(x[j], g) ? 1u : 0u) << j;
                    part <<= kV * (lane % kWordLanes);
#pragma unroll
                    for (int d = 1; d < kWordLanes; d <<= 1) part |= __shfl_xor_sync(FULL, part, d);
                    // the load's words sit in groups of kWordLanes lanes; word kV (h + k) + i
                    // belongs to lane kV (h + k) + i, group i holds it
                    const uint32_t mine = __shfl_sync(FULL, part, kWordLanes * (lane % kV));
                    if (lane / kV == h + k) word = mine;
                }
            }
        } else {
            T v[W];
#pragma unroll
            for (int i = 0; i < W; ++i) v[i] = col[base + 32 * i + lane];
#pragma unroll
            for (int i = 0; i < W; ++i) {
                const uint32_t m = __ballot_sync(FULL, passes(v[i], g));
                if (lane == i) word = m;
            }
        }
    } else {
        for (int i = 0; i < W; ++i) {
            const int64_t r = base + 32 * i + lane;
            const uint32_t m = __ballot_sync(FULL, r < n && passes(col[r < n ? r : 0], g));
            if (lane == i) word = m;
        }
    }
    return word;
}

// Rows the predicate reads: none when no value passes.
template <typename T>
__device__ __forceinline__ int64_t live_rows(const int64_t* d_nrows, int64_t ncap, const Range<T>& g) {
    return g.none ? 0 : actual_rows(d_nrows, ncap);
}

// tile_cnt[tile]: passing rows of the tile; bits: one word per 32 rows (null: not kept).
template <typename T, int W>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
filter_count_kernel(const T* __restrict__ col, int64_t ncap, const int64_t* __restrict__ d_nrows, Range<T> g,
                    int64_t ntiles, int32_t* __restrict__ tile_cnt, uint32_t* __restrict__ bits) {
    constexpr int kTile = kWarps * 32 * W;
    __shared__ int32_t s_warp[2][kWarps];
    allow_dependents();
    const int64_t n = live_rows(d_nrows, ncap, g);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int flip = 0;  // one barrier per tile: the warps' counts alternate between two rows
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, flip ^= 1) {
        const int64_t base = tile * kTile + warp * (32 * W);
        uint32_t word = 0;
        if (base < n) {
            word = warp_words<T, W>(col, base, n, g, lane);
            if (bits && lane < W) bits[base / 32 + lane] = word;
        }
        const uint32_t c = __reduce_add_sync(FULL, static_cast<uint32_t>(__popc(word)));
        if (lane == 0) s_warp[flip][warp] = static_cast<int32_t>(c);
        __syncthreads();
        if (threadIdx.x == 0) {
            int32_t t = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) t += s_warp[flip][w];
            tile_cnt[tile] = t;
        }
    }
}

template <typename T, int W>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
filter_write_kernel(const T* __restrict__ col, int64_t ncap, const int64_t* __restrict__ d_nrows, Range<T> g,
                    int64_t ntiles, const int32_t* tile_cnt, const uint32_t* bits, int32_t* __restrict__ sel,
                    int64_t* __restrict__ d_nsel) {
    constexpr int kTile = kWarps * 32 * W;
    __shared__ uint32_t s_warp[2][kWarps];
    __shared__ int32_t s_rows[W == 32 ? kWarps : 1][W == 32 ? kStage : 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // this block's tiles: an even split
    const int64_t G = gridDim.x, b = blockIdx.x;
    const int t0 = static_cast<int>(ntiles * b / G), t1 = static_cast<int>(ntiles * (b + 1) / G);
    wait_prior();  // the counts and bits
    const int64_t n = live_rows(d_nrows, ncap, g);
    uint32_t before = 0;  // passing rows of the tiles before this block's (they fit int32: nrows < 2^31)
    const int4* cnt4 = reinterpret_cast<const int4*>(tile_cnt);
#pragma unroll 8
    for (int k = threadIdx.x; k < t0 / 4; k += kThreads) {
        const int4 x = cnt4[k];
        before += static_cast<uint32_t>(x.x + x.y + x.z + x.w);
    }
    if (threadIdx.x < (t0 & 3)) before += static_cast<uint32_t>(tile_cnt[(t0 & ~3) + threadIdx.x]);
    before = __reduce_add_sync(FULL, before);
    if (lane == 0) s_warp[1][warp] = before;
    __syncthreads();
    uint32_t pos = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) pos += s_warp[1][w];
    const uint32_t lt = lanemask_lt();
    int flip = 0;  // as in the count
    for (int tile = t0; tile < t1; ++tile, flip ^= 1) {
        const int64_t base = static_cast<int64_t>(tile) * kTile + warp * (32 * W);
        uint32_t word = 0;
        if (base < n) {
            if (bits) word = lane < W ? bits[base / 32 + lane] : 0;
            else word = warp_words<T, W>(col, base, n, g, lane);
        }
        const uint32_t c = __popc(word);
        const uint32_t incl = warp_incl_scan(c);
        if (lane == 31) s_warp[flip][warp] = incl;
        __syncthreads();
        uint32_t at = pos + incl - c;  // output slot of the lane's first row
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t x = s_warp[flip][w];
            if (w < warp) at += x;
            pos += x;
        }
        const uint32_t total = __shfl_sync(FULL, incl, 31);
        if (W == 32 && total < kDense) {
            // Each lane appends its word's rows to the warp's stage, which then goes out
            // in whole coalesced stores (one row in 33 words apart, so lanes with equal
            // counts hit different banks).
            const uint32_t first = __shfl_sync(FULL, at, 0);
            int32_t* stage = s_rows[warp];
            uint32_t p = incl - c;
            const int32_t row = static_cast<int32_t>(base) + 32 * lane;
#pragma unroll
            for (int bit = 0; bit < 32; ++bit)
                if ((word >> bit) & 1u) {
                    stage[p + (p >> 5)] = row + bit;
                    ++p;
                }
            __syncwarp();
            for (uint32_t k = lane; k < total; k += 32) sel[first + k] = stage[k + (k >> 5)];
        } else {
            const uint32_t row = static_cast<uint32_t>(base) + lane;
#pragma unroll 8
            for (int i = 0; i < W; ++i) {
                const uint32_t m = __shfl_sync(FULL, word, i);
                const uint32_t p = __shfl_sync(FULL, at, i);
                if ((m >> lane) & 1u) sel[p + __popc(m & lt)] = static_cast<int32_t>(row + 32 * i);
            }
        }
    }
    if (b == G - 1 && threadIdx.x == 0) *d_nsel = static_cast<int64_t>(pos);
}

constexpr int64_t kNarrowTiles = 2048;  // narrow tiles at most, whatever the chip

// Scratch: a count per tile, then the bits (when kept), one word per 32 rows, whole
// tiles.
size_t count_bytes(int64_t nrows) {
    const int64_t wide = cdiv(nrows, kWarps * 32 * kWide);
    const int64_t narrow = std::min(cdiv(nrows, kWarps * 32 * kNarrow), kNarrowTiles);
    return align_up(static_cast<size_t>(std::max(wide, narrow)) * 4, 256);
}
size_t bits_bytes(int64_t nrows) { return static_cast<size_t>(cdiv(nrows, kWarps * 32 * kWide)) * (kWarps * kWide * 4); }

template <typename T, int W>
void launch_filter_w(const T* col, int64_t nrows, const int64_t* d_nrows, const Range<T>& g, int64_t max_blocks,
                     int32_t* d_sel, int64_t* d_nsel, int32_t* cnt, uint32_t* bits, cudaStream_t st) {
    const int64_t ntiles = cdiv(nrows, kWarps * 32 * W);
    const dim3 grid(static_cast<unsigned>(std::min(ntiles, max_blocks)));
    filter_count_kernel<T, W><<<grid, kThreads, 0, st>>>(col, nrows, d_nrows, g, ntiles, cnt, bits);
    launch_after(filter_write_kernel<T, W>, grid, dim3(kThreads), 0, st, col, nrows, d_nrows, g, ntiles, cnt, bits,
                 d_sel, d_nsel);
}

template <typename T>
void launch_filter(const void* col, int64_t nrows, const int64_t* d_nrows, int64_t lo, int64_t hi, int32_t* d_sel,
                   int64_t* d_nsel, int32_t* cnt, uint32_t* bits, cudaStream_t st) {
    const T* c = static_cast<const T*>(col);
    const Range<T> g = make_range<T>(lo, hi);
    // one wave of the chip holds every block
    const int64_t max_blocks = static_cast<int64_t>(sm_count()) * kBlocksPerSm;
    if (cdiv(nrows, kWarps * 32 * kNarrow) <= std::min(max_blocks, kNarrowTiles))
        launch_filter_w<T, kNarrow>(c, nrows, d_nrows, g, max_blocks, d_sel, d_nsel, cnt, bits, st);
    else
        launch_filter_w<T, kWide>(c, nrows, d_nrows, g, max_blocks, d_sel, d_nsel, cnt, bits, st);
}

// cnt: count_bytes(nrows) of device scratch; bits: bits_bytes(nrows), or null.
void launch_filter_type(int32_t type, const void* col, int64_t nrows, const int64_t* d_nrows, int64_t lo, int64_t hi,
                        int32_t* d_sel, int64_t* d_nsel, int32_t* cnt, uint32_t* bits, cudaStream_t st) {
    switch (type) {
        case PX_I8: launch_filter<int8_t>(col, nrows, d_nrows, lo, hi, d_sel, d_nsel, cnt, bits, st); break;
        case PX_I32: launch_filter<int32_t>(col, nrows, d_nrows, lo, hi, d_sel, d_nsel, cnt, bits, st); break;
        default: launch_filter<int64_t>(col, nrows, d_nrows, lo, hi, d_sel, d_nsel, cnt, bits, st); break;
    }
    note_launch();
    note_launch();
}

}  // namespace
}  // namespace px

using namespace px;

extern "C" {

size_t px_filter_ws_bytes(int64_t nrows) {
    if (nrows < 0) nrows = 0;
    return kWsScratch + count_bytes(nrows) + align_up(bits_bytes(nrows), 256);
}

px_status px_filter(const px_col* col, int64_t nrows, const int64_t* d_nrows, int64_t lo, int64_t hi,
                    int32_t* d_sel, int64_t* d_nsel, void* d_ws, size_t ws_bytes, void* stream) {
    CallRange nvtx_range("px_filter");
    set_error("");
    px_status s = check_col(col, "px_filter col", nrows == 0);
    if (s != PX_OK) return s;
    if (nrows < 0 || nrows > INT32_MAX)
        return fail(PX_ERR_UNSUPPORTED, "px_filter: nrows %lld outside [0, 2^31)", (long long)nrows);
    if (!d_sel || !d_nsel) return fail(PX_ERR_INVALID, "px_filter: null d_sel or d_nsel");
    s = check_ws(d_ws, ws_bytes, px_filter_ws_bytes(nrows), "px_filter");
    if (s != PX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (nrows == 0) {
        cudaMemsetAsync(d_nsel, 0, sizeof(int64_t), st);
        return check_launch("px_filter");
    }
    char* scratch = static_cast<char*>(d_ws) + kWsScratch;
    launch_filter_type(col->type, col->data, nrows, d_nrows, lo, hi, d_sel, d_nsel, reinterpret_cast<int32_t*>(scratch),
                       reinterpret_cast<uint32_t*>(scratch + count_bytes(nrows)), st);
    return check_launch("px_filter");
}

}  // extern "C"

// ---------------------------------------------------------------------------
// px_filter_noalloc: the same filter for callers that cannot allocate device
// memory, so cannot provide a workspace: e.g. code running under a host engine
// whose memory manager owns every device byte and forbids side allocations, or a
// serving loop that reserves all memory at start-up and must not call cudaMalloc
// (which can synchronise the device) on its hot path. Its scratch (the counts, after
// a header kept for the workspace layout the filter kernels share) lives in the
// file-scope device array below instead of a caller workspace; it is too small for
// one bit per row, so the write pass reads the column again.
namespace px {
namespace {

// Header (status word) and room for the counts (no bits are kept).
constexpr size_t kNoallocScratchBytes = 262400;  // the documented size
static_assert(kWsScratch + PX_FILTER_NOALLOC_MAX_ROWS / (kWarps * 32 * kWide) * 4 <= kNoallocScratchBytes,
              "the counts fit the static scratch");

// Held by every GPU that loads the library, until the process exits.
static __device__ __align__(256) unsigned char g_filter_scratch[kNoallocScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
void* g_noalloc_addr[kMaxDevices] = {};

// Device address of g_filter_scratch on the current device. In host code the
// array's name is only a host-side stand-in, so the address is looked up once per
// device with cudaGetSymbolAddress (with that device current) and cached.
px_status noalloc_scratch(void** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(PX_ERR_CUDA, "px_filter_noalloc: cudaGetDevice: %s", cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return fail(PX_ERR_UNSUPPORTED, "px_filter_noalloc: device %d", dev);
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_filter_scratch);
        if (e != cudaSuccess || !p)
            return fail(PX_ERR_CUDA, "px_filter_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
        g_noalloc_addr[dev] = p;
    }
    *out = g_noalloc_addr[dev];
    return PX_OK;
}

}  // namespace
}  // namespace px

extern "C" px_status px_filter_noalloc(const px_col* col, int64_t nrows, const int64_t* d_nrows, int64_t lo,
                                       int64_t hi, int32_t* d_sel, int64_t* d_nsel, int32_t* d_status,
                                       void* stream) {
    CallRange nvtx_range("px_filter_noalloc");
    set_error("");
    px_status s = check_col(col, "px_filter_noalloc col", nrows == 0);
    if (s != PX_OK) return s;
    if (nrows < 0 || nrows > PX_FILTER_NOALLOC_MAX_ROWS)
        return fail(PX_ERR_UNSUPPORTED, "px_filter_noalloc: nrows %lld outside [0, %lld]; use px_filter",
                    (long long)nrows, (long long)PX_FILTER_NOALLOC_MAX_ROWS);
    if (!d_sel || !d_nsel) return fail(PX_ERR_INVALID, "px_filter_noalloc: null d_sel or d_nsel");
    void* scratch = nullptr;
    if ((s = noalloc_scratch(&scratch)) != PX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // The array keeps whatever the previous call left there; every count a call
    // uses is written before it is read, so nothing needs clearing. The filter
    // records no data-dependent error, so the status is always PX_OK.
    if (nrows == 0) {
        cudaMemsetAsync(d_nsel, 0, sizeof(int64_t), st);
    } else {
        int32_t* cnt = reinterpret_cast<int32_t*>(static_cast<char*>(scratch) + kWsScratch);
        launch_filter_type(col->type, col->data, nrows, d_nrows, lo, hi, d_sel, d_nsel, cnt, nullptr, st);
    }
    if (d_status) cudaMemsetAsync(d_status, 0, sizeof(int32_t), st);
    return check_launch("px_filter_noalloc");
}

// px_fragments_run: a batch of independent plan fragments, each FilterProject ->
// join probe -> HashAggregation (Single mode) over one probe batch and one
// prebuilt dimension table (the operators of Sec. 3.2 and the join probe
// pipeline of Sec. 3.1), run as ONE persistent fused kernel plus one emit kernel.
// The paper finds small vectors leave a GPU underused (Sec. 3.3.2) and results
// sensitive to batch size (Sec. 3.4); batching whole fragments into one launch is
// this library's answer for many small fragments.
//
// Work items are (fragment, chunk of rows), handed out by a device counter in
// the order of decreasing fragment size. Every warp of a block walks its own runs of
// 128 rows of the chunk: it reads the filter column and the join keys (4 consecutive
// rows per lane, vector loads) and appends the passing rows and their keys to a queue in
// shared memory; whenever the queue holds 32 x ITEMS rows the warp takes them off, every
// lane with ITEMS rows: their home buckets (one sector: keys, build rows
// and, when the dimension was built with its group column copied, the group keys;
// else the group key is gathered from the build column at the build row) with the
// aggregate inputs loading beside them; the aggregates go into the fragment's dense
// accumulators (group key - group_lo indexes them):
//   * shared mode (small key ranges): block arrays in shared memory, cleared per
//     work item and added into the fragment's global arrays at its end;
//   * direct mode: 64-bit reductions straight into the global arrays.
// The emit kernel compacts each fragment's occupied slots into its output in
// key order (single pass, per-fragment bounded look-back).
//
// What bounds it: the lookups' dependent round trips (filter and key, bucket, now and
// then the next bucket) at 32 warps per SM, then DRAM (56 % busy): 512
// fragments, 388M rows, 28 B per row of columns and 2.4 GB of tables. Measured on
// that batch: every row looked up in place 12.8 ms; passing rows queued and looked up
// by full warps 6.0 ms; the next run's columns prefetched into L2, the items' walks
// merged and block arrays of 24 KB 3.8 ms; spread tables, items of 32768 rows and the keys
// read beside the filter 3.5 ms (3.4 TB/s). Blocks of 512 threads with 2 rows in flight
// per thread (two per SM, 64 registers, of which three aggregates spill 124 bytes and four
// 312): 3.5 ms; 256 x 2 3.9 ms, 512 x 4 (one per SM, 128 registers, no spills up to three
// aggregates) 3.8 ms.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "px_common.cuh"
#include "px_table.cuh"

namespace px {
namespace {

// Shared-mode block accumulators, direct mode above. 48M rows over 500,000-key tables, a
// 30 % filter, 3 aggregates (24 bytes a group), uniform keys / Zipf(1.1) keys, us: 1100 groups
// shared 494 / 410, direct 733 / 956; 2000 groups 557 / 448 and 673 / 934; 2700 groups (63 KB)
// 834 / 622 and 661 / 878; 4000 groups (94 KB) 682 / 645 and 643 / 957. Direct reductions of a
// hot group queue at one address; large arrays leave every fragment of the batch less L1:
// with the queues, two blocks of up to 42 KB fit the 164 KB split of the SM's memory
// (512 fragments: 24 KB 3.48 ms, 40 KB 3.45, 48 KB 3.70).
// Arrays of more than kSmallAcc bytes only where a work item has many rows per group to clear
// and flush them for: 207 small fragments (500 to 200,000 rows) 113.7 us without, 115.6 with.
constexpr size_t kSmemAccBudget = 42 * 1024;
constexpr size_t kSmallAcc = 24 * 1024;
constexpr int64_t kMaxChunk = 32768;               // rows per work item, unless the caller says (65536: 3 % slower)
constexpr uint64_t kRepSlots = 1024;               // shared-mode slots with their replicas, at most
constexpr int kEmitThreads = 256;
constexpr int kEmitItems = 8;
constexpr int kEmitTile = kEmitThreads * kEmitItems;
constexpr int kMajority = 6;  // smallest lane group worth a warp reduction

// Device plan of one fragment.
struct FragDev {
    const int64_t* key;
    const void* filter;
    int64_t lo, hi;
    int64_t nrows;
    // aggregate k reads column pa[k] (width wa[k]) and, for SUM_MUL, pb[k] (wb[k])
    const void* pa[PX_FRAG_MAX_AGGS];
    const void* pb[PX_FRAG_MAX_AGGS];
    int32_t same[PX_FRAG_MAX_AGGS];  // an earlier SUM of the column pa[k], whose value is reused, or -1
    int32_t op[PX_FRAG_MAX_AGGS], wa[PX_FRAG_MAX_AGGS], wb[PX_FRAG_MAX_AGGS];
    // the distinct columns a row is read from (filter, key, aggregate inputs)
    int32_t nstream;
    int32_t stream_w[PX_FRAG_MAX_COLS + 2];
    const void* stream[PX_FRAG_MAX_COLS + 2];
    int32_t filter_w, naggs, group_w, count_agg;  // count_agg: a COUNT aggregate, or -1
    TableView t;
    int64_t nbuild;
    const void* group;
    int64_t group_lo;
    uint32_t D;      // dense slots
    int32_t shared;  // 1: block accumulators in shared memory
    uint32_t rep_shift;  // shared mode: 1 << rep_shift replicas of every slot, side by side
    uint32_t reserved;
    int64_t chunk;   // rows per work item
    unsigned long long* acc;  // [naggs][D]
    uint8_t* occ;             // [D] occupancy flags (only without COUNT)
    uint64_t* emit_states;    // look-back states of the fragment's emit tiles
    void* out_keys;
    int64_t* out_aggs[PX_FRAG_MAX_AGGS];
    int64_t* ngroups;
    int64_t max_groups;
};

struct PlanHeader {
    int32_t nfrags;
    int32_t reserved;
    int64_t nitems;  // work items
    int64_t nemit;   // emit tiles
    int64_t pad[5];
};

// Plan (host staging and its device copy): header, item_start[nfrags + 1],
// emit_start[nfrags + 1], FragDev[nfrags]; fragments in work order.
struct PlanLayout {
    size_t items, emits, frags, total;
};
PlanLayout plan_layout(int32_t n) {
    PlanLayout L;
    L.items = sizeof(PlanHeader);
    L.emits = L.items + align_up(8 * static_cast<size_t>(n + 1), 64);
    L.frags = L.emits + align_up(8 * static_cast<size_t>(n + 1), 64);
    L.total = L.frags + align_up(sizeof(FragDev) * static_cast<size_t>(n), 64);
    return L;
}

// Largest p with start[p] <= x (start ascending, start[0] = 0 <= x).
__device__ __forceinline__ int find_frag(const int64_t* start, int n, int64_t x) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (start[mid] <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int64_t load_w(const void* p, int w, int64_t i) { return load_int(p, w, i); }

// Adds x (mod 2^64) to a 64-bit value held as 32-bit words lo/hi in shared memory.
__device__ __forceinline__ void add_split(uint32_t* lo, uint32_t* hi, uint64_t x) {
    const uint32_t xl = static_cast<uint32_t>(x), xh = static_cast<uint32_t>(x >> 32);
    const uint32_t old = atomicAdd(lo, xl);
    const uint32_t add_hi = xh + (old + xl < old ? 1u : 0u);
    if (add_hi) red_add_shared(hi, add_hi);
}

constexpr int kFilterRows = 4;                  // consecutive rows a lane filters at a time
constexpr int kWarpRows = 32 * kFilterRows;     // rows a warp filters at a time
constexpr uint32_t kNone = 0xffffffffu;         // no dense slot

// Rows a warp's queue holds at most: one short of a full take, plus one filter step.
template <int ITEMS>
constexpr int kQueue = 32 * ITEMS - 1 + kWarpRows;

// Bit j of the result: row r + j passes lo <= col < hi. A full run of kFilterRows
// rows below r1 is one aligned vector load (r is a multiple of kFilterRows and the
// column is 16-byte aligned).
template <typename T>
__device__ __forceinline__ uint32_t filter_rows(const T* col, int64_t lo, int64_t hi, int64_t r, int64_t r1) {
    T v[kFilterRows];
    uint32_t ok = 0;
    if (r + kFilterRows <= r1) {
        if (sizeof(T) == 8) {
            const longlong2 x = *reinterpret_cast<const longlong2*>(col + r);
            const longlong2 y = *reinterpret_cast<const longlong2*>(col + r + 2);
            v[0] = static_cast<T>(x.x);
            v[1] = static_cast<T>(x.y);
            v[2] = static_cast<T>(y.x);
            v[3] = static_cast<T>(y.y);
        } else if (sizeof(T) == 4) {
            const int4 x = *reinterpret_cast<const int4*>(col + r);
            v[0] = static_cast<T>(x.x);
            v[1] = static_cast<T>(x.y);
            v[2] = static_cast<T>(x.z);
            v[3] = static_cast<T>(x.w);
        } else {
            const char4 x = *reinterpret_cast<const char4*>(col + r);
            v[0] = static_cast<T>(x.x);
            v[1] = static_cast<T>(x.y);
            v[2] = static_cast<T>(x.z);
            v[3] = static_cast<T>(x.w);
        }
#pragma unroll
        for (int j = 0; j < kFilterRows; ++j)
            ok |= (static_cast<int64_t>(v[j]) >= lo && static_cast<int64_t>(v[j]) < hi ? 1u : 0u) << j;
    } else {
#pragma unroll
        for (int j = 0; j < kFilterRows; ++j)
            if (r + j < r1) {
                const int64_t x = static_cast<int64_t>(col[r + j]);
                ok |= (x >= lo && x < hi ? 1u : 0u) << j;
            }
    }
    return ok;
}

// Rows [r0, r1) of fragment f (r0 a multiple of kFilterRows). SHARED: accumulate
// into the block arrays lo/hi ([naggs][D][replicas] each) and occupancy bits; else
// reduce into the global arrays. `queue`: this warp's kQueue<ITEMS> entries.
// Only rows that pass the filter touch the value and table memory, and every
// lane of a lookup holds one: with the lookups predicated in place a filter that
// keeps 30 % of the rows left two lanes of three idle through them (ncu: 19.5
// threads per instruction).
// W8: every aggregated column of the batch is 8 bytes wide (no width switches).
template <int THREADS, int ITEMS, int NA, bool W8, bool SHARED>
__device__ void frag_rows(const FragDev& f, int64_t r0, int64_t r1, uint32_t* s_lo, uint32_t* s_hi,
                          uint32_t* s_occ, int64_t* queue_key, uint32_t* queue, int32_t* status) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t nb = static_cast<uint32_t>(table_buckets(f.t.hdr->nbuild, 1, f.t.hdr->spread));
    // the group column copied into the table at build time: read with the key
    const bool group_in_table = f.t.hdr->pay_src == f.group && f.t.hdr->pay_w == f.group_w;
    const int naggs = f.naggs;
    const uint32_t lt = lanemask_lt();
    const uint32_t rep = SHARED ? static_cast<uint32_t>(lane) & ((1u << f.rep_shift) - 1) : 0;
    uint32_t held = 0;  // rows in the queue

    // Takes the last `n` (1..32 * ITEMS) rows off the queue and aggregates them.
    auto take = [&](uint32_t n) {
        uint32_t row[ITEMS];
        int64_t key[ITEMS], v[NA][ITEMS];
        BucketRegs bv[ITEMS];
        uint32_t hb[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const uint32_t e = 32 * i + lane;
            row[i] = e < n ? queue[held - n + e] : kNone;
            key[i] = e < n ? queue_key[held - n + e] : kEmpty;
        }
        __syncwarp();  // the entries are read: the next append may overwrite them
        held -= n;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            hb[i] = home_bucket(static_cast<uint64_t>(key[i]), nb);
            bv[i] = load_bucket(f.t.bk + hb[i]);  // hb < nb: inside the table
        }
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            if (a >= naggs) break;
            if (f.op[a] == PX_COUNT) continue;
            const int same = f.same[a];
            if (same >= 0) {
#pragma unroll
                for (int b = 0; b < a; ++b)
                    if (same == b) {
#pragma unroll
                        for (int i = 0; i < ITEMS; ++i) v[a][i] = v[b][i];
                    }
            } else {
#pragma unroll
                for (int i = 0; i < ITEMS; ++i)
                    v[a][i] = row[i] != kNone ? load_w(f.pa[a], W8 ? 8 : f.wa[a], r0 + row[i]) : 0;
            }
            if (f.op[a] == PX_SUM_MUL) {
#pragma unroll
                for (int i = 0; i < ITEMS; ++i)
                    if (row[i] != kNone)
                        v[a][i] = static_cast<int64_t>(static_cast<uint64_t>(v[a][i]) *
                                                       static_cast<uint64_t>(load_w(f.pb[a], W8 ? 8 : f.wb[a], r0 + row[i])));
            }
        }
        // The match of every item; the keys displaced past their home bucket (about one
        // in eight, so some lane of nearly every warp) then walk on together, one round
        // trip for all of the warp's items.
        int32_t mrow[ITEMS], mpay[ITEMS];
        uint32_t pend = 0;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            mrow[i] = -1;
            mpay[i] = 0;
            if (key[i] == kEmpty) continue;
            bool end;
            const int l = bucket_find(bv[i], key[i], &end);
            if (l >= 0) {
                mrow[i] = bucket_row(bv[i], l);
                mpay[i] = bucket_pay(bv[i], l);
            } else if (!end) {
                pend |= 1u << i;
            }
        }
        for (uint32_t round = 1; round < nb && pend; ++round) {
#pragma unroll
            for (int i = 0; i < ITEMS; ++i)
                if ((pend >> i) & 1u) {
                    hb[i] = hb[i] + 1 == nb ? 0 : hb[i] + 1;
                    bv[i] = load_bucket(f.t.bk + hb[i]);
                }
#pragma unroll
            for (int i = 0; i < ITEMS; ++i)
                if ((pend >> i) & 1u) {
                    bool end;
                    const int l = bucket_find(bv[i], key[i], &end);
                    if (l >= 0) {
                        mrow[i] = bucket_row(bv[i], l);
                        mpay[i] = bucket_pay(bv[i], l);
                    }
                    if (l >= 0 || end) pend &= ~(1u << i);
                }
        }
        __syncwarp();
        uint32_t slot[ITEMS];  // dense slot of the row's group, or kNone
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            slot[i] = kNone;
            if (mrow[i] < 0) continue;
            const int64_t gk = group_in_table ? static_cast<int64_t>(mpay[i]) : load_w(f.group, f.group_w, mrow[i]);
            const uint64_t d = static_cast<uint64_t>(gk - f.group_lo);
            if (d < f.D) slot[i] = static_cast<uint32_t>(d);
            else set_status(status, PX_ERR_UNSUPPORTED);
        }
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            // Rows sharing lane 0's slot: summed across the warp, applied once by lane 0
            // (not where every lane has a replica of its own).
            uint32_t apply = slot[i];
            uint32_t cnt = 1;
            if (!SHARED || f.rep_shift < 5) {
                const uint32_t c0 = __shfl_sync(FULL, slot[i], 0);
                const uint32_t mm = __ballot_sync(FULL, slot[i] == c0);
                if (c0 != kNone && __popc(mm) >= kMajority) {
                    const bool in = (mm >> lane) & 1u;
#pragma unroll
                    for (int a = 0; a < NA; ++a) {
                        if (a >= naggs) break;
                        if (f.op[a] == PX_COUNT) continue;
                        const uint64_t x = warp_sum_u64(in ? static_cast<uint64_t>(v[a][i]) : 0);
                        if (lane == 0) v[a][i] = static_cast<int64_t>(x);
                    }
                    if (lane == 0) cnt = __popc(mm);
                    else if (in) apply = kNone;
                }
            }
            if (apply == kNone) continue;
            if (SHARED) {
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    if (a >= naggs) break;
                    const uint32_t o = ((static_cast<uint32_t>(a) * f.D + apply) << f.rep_shift) + rep;
                    // a work item counts fewer than 2^32 rows
                    if (f.op[a] == PX_COUNT) red_add_shared(&s_lo[o], cnt);
                    else add_split(&s_lo[o], &s_hi[o], static_cast<uint64_t>(v[a][i]));
                }
                if (f.count_agg < 0) red_or_shared(&s_occ[apply / 32], 1u << (apply % 32));
            } else {
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    if (a >= naggs) break;
                    red_add_global(&f.acc[static_cast<size_t>(a) * f.D + apply],
                                   f.op[a] == PX_COUNT ? cnt : static_cast<unsigned long long>(v[a][i]));
                }
                if (f.count_agg < 0) f.occ[apply] = 1;  // every writer stores the same value
            }
        }
    };

    for (int64_t tb = r0 + warp * kWarpRows;; tb += THREADS * kFilterRows) {
        const bool more = tb < r1;
        if (more) {
            // The next run's columns start on their way to L2 while this one is
            // aggregated (one bulk prefetch per column, lanes 0..ncols+1).
            const int64_t nt = tb + THREADS * kFilterRows;
            if (lane < f.nstream && nt < r1) {
                const int64_t w = f.stream_w[lane];
                const int64_t bytes = ((r1 - nt < kWarpRows ? r1 - nt : kWarpRows) * w) & ~int64_t(15);
                if (bytes) prefetch_l2(static_cast<const char*>(f.stream[lane]) + nt * w, static_cast<uint32_t>(bytes));
            }
            // The keys are read beside the filter column (their sectors are needed for one
            // passing row in four anyway), so a lookup waits for its bucket alone.
            const int64_t r = tb + kFilterRows * lane;
            int64_t k[kFilterRows];
            if (r + kFilterRows <= r1) {
#pragma unroll
                for (int j = 0; j < kFilterRows; j += 2) {
                    const longlong2 x = *reinterpret_cast<const longlong2*>(f.key + r + j);
                    k[j] = x.x;
                    k[j + 1] = x.y;
                }
            } else {
#pragma unroll
                for (int j = 0; j < kFilterRows; ++j) k[j] = r + j < r1 ? f.key[r + j] : kEmpty;
            }
            uint32_t ok;
            if (!f.filter) {
                ok = r + kFilterRows <= r1 ? (1u << kFilterRows) - 1 : (r < r1 ? (1u << (r1 - r)) - 1 : 0);
            } else if (f.filter_w == 4) {
                ok = filter_rows(static_cast<const int32_t*>(f.filter), f.lo, f.hi, r, r1);
            } else if (f.filter_w == 8) {
                ok = filter_rows(static_cast<const int64_t*>(f.filter), f.lo, f.hi, r, r1);
            } else {
                ok = filter_rows(static_cast<const int8_t*>(f.filter), f.lo, f.hi, r, r1);
            }
            const uint32_t rel = static_cast<uint32_t>(r - r0);
#pragma unroll
            for (int j = 0; j < kFilterRows; ++j) {
                const bool p = (ok >> j) & 1u;
                const uint32_t m = __ballot_sync(FULL, p);
                if (p) {
                    queue[held + __popc(m & lt)] = rel + j;
                    queue_key[held + __popc(m & lt)] = k[j];
                }
                held += __popc(m);
            }
            __syncwarp();
        }
        // Full takes while rows are left to filter, whatever is held at the end.
        while (held >= (more ? 32u * ITEMS : 1u)) take(held < 32u * ITEMS ? held : 32u * ITEMS);
        if (!more) break;
    }
}

// Persistent fused kernel: (fragment, chunk) work items from a device counter.
template <int THREADS, int ITEMS, int NA, bool W8>
__global__ void __launch_bounds__(THREADS, (ITEMS > 2 ? 512 : 1024) / THREADS)
frag_kernel(const PlanHeader* __restrict__ ph, const int64_t* __restrict__ item_start, const FragDev* __restrict__ fd,
            unsigned long long* counter, int32_t* status) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int64_t s_item;
    __shared__ int32_t s_p;
    // The work item's fragment plan, copied to shared memory once per item: the
    // reductions' memory clobbers would otherwise reload its fields from global
    // memory after every update.
    __shared__ __align__(16) FragDev s_f;
    __shared__ int64_t s_queue_key[THREADS / 32][kQueue<ITEMS>];
    __shared__ uint32_t s_queue[THREADS / 32][kQueue<ITEMS>];
    int64_t* queue_key = s_queue_key[threadIdx.x >> 5];
    uint32_t* queue = s_queue[threadIdx.x >> 5];
    const int n = ph->nfrags;
    const int64_t nitems = ph->nitems;
    for (;;) {
        if (threadIdx.x == 0) {
            const int64_t it = static_cast<int64_t>(atomicAdd(counter, 1ull));
            s_item = it;
            s_p = it < nitems ? find_frag(item_start, n, it) : 0;
        }
        __syncthreads();
        const int64_t item = s_item;
        const int p = s_p;
        if (item < nitems) {
            const uint32_t* src = reinterpret_cast<const uint32_t*>(&fd[p]);
            uint32_t* dst = reinterpret_cast<uint32_t*>(&s_f);
            for (int w = threadIdx.x; w < static_cast<int>(sizeof(FragDev) / 4); w += THREADS) dst[w] = src[w];
        }
        __syncthreads();
        if (item >= nitems) break;
        const FragDev& f = s_f;
        // A table this fragment cannot use: its rows are skipped.
        if (f.t.hdr->magic != kMagic || f.t.hdr->nsegs != 1 || f.t.hdr->unique == 0 || f.t.hdr->nbuild > f.nbuild) {
            if (threadIdx.x == 0) set_status(status, PX_ERR_INVALID);
            continue;
        }
        const int64_t r0 = (item - item_start[p]) * f.chunk;
        const int64_t r1 = r0 + f.chunk < f.nrows ? r0 + f.chunk : f.nrows;
        if (!f.shared) {
            frag_rows<THREADS, ITEMS, NA, W8, false>(f, r0, r1, nullptr, nullptr, nullptr, queue_key, queue, status);
            continue;
        }
        const uint32_t D = f.D;
        const int naggs = f.naggs;
        const uint32_t rs = f.rep_shift;
        const uint32_t slots = (naggs * D) << rs;
        uint32_t* s_lo = reinterpret_cast<uint32_t*>(smem);
        uint32_t* s_hi = s_lo + slots;
        uint32_t* s_occ = s_hi + slots;
        const uint32_t words = 2 * slots + (f.count_agg < 0 ? (D + 31) / 32 : 0);
        for (uint32_t w = threadIdx.x; w < words; w += THREADS) s_lo[w] = 0;
        __syncthreads();
        frag_rows<THREADS, ITEMS, NA, W8, true>(f, r0, r1, s_lo, s_hi, s_occ, queue_key, queue, status);
        __syncthreads();
        const uint32_t reps = 1u << rs;
        for (uint32_t o = threadIdx.x; o < naggs * D; o += THREADS) {
            uint64_t x = 0;
            for (uint32_t k = 0; k < reps; ++k) {
                const uint32_t w = (o << rs) + ((k + threadIdx.x) & (reps - 1));  // banks spread over the threads
                x += (static_cast<uint64_t>(s_hi[w]) << 32) | s_lo[w];
            }
            if (x) red_add_global(&f.acc[o], x);
        }
        if (f.count_agg < 0)
            for (uint32_t d = threadIdx.x; d < D; d += THREADS)
                if ((s_occ[d / 32] >> (d % 32)) & 1u) f.occ[d] = 1;
        // The next item's clear waits for every thread's flush at the loop top.
    }
}

// Writes each fragment's occupied slots as output groups in key order.
__global__ void __launch_bounds__(kEmitThreads)
frag_emit_kernel(const PlanHeader* __restrict__ ph, const int64_t* __restrict__ emit_start,
                 const FragDev* __restrict__ fd, unsigned long long* counter, int32_t* status) {
    __shared__ int64_t s_tile;
    __shared__ int64_t s_excl;
    __shared__ int32_t s_warp[kEmitThreads / 32];
    wait_prior();  // the accumulators (and the plan)
    const int64_t tile = next_tile(counter, &s_tile);
    // The fragment's plan, copied once: its fields would be loaded again, each a memory
    // round trip, after every ordered access below.
    __shared__ __align__(16) FragDev s_f;
    const int p = find_frag(emit_start, ph->nfrags, tile);
    for (int w = threadIdx.x; w < static_cast<int>(sizeof(FragDev) / 4); w += kEmitThreads)
        reinterpret_cast<uint32_t*>(&s_f)[w] = reinterpret_cast<const uint32_t*>(&fd[p])[w];
    __syncthreads();
    const FragDev& f = s_f;
    const int64_t lt = tile - emit_start[p];  // tile within the fragment
    const int64_t ntiles = emit_start[p + 1] - emit_start[p];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t base = lt * kEmitTile + warp * (32 * kEmitItems);
    const int64_t D = f.D;
    uint32_t mask[kEmitItems];
    int32_t cnt = 0;
#pragma unroll
    for (int i = 0; i < kEmitItems; ++i) {
        const int64_t e = base + i * 32 + lane;
        bool occ = false;
        if (e < D) occ = f.count_agg >= 0 ? f.acc[f.count_agg * D + e] != 0 : f.occ[e] != 0;
        mask[i] = __ballot_sync(FULL, occ);
        cnt += __popc(mask[i]);
    }
    if (lane == 0) s_warp[warp] = cnt;
    __syncthreads();
    if (warp == 0) {
        const int32_t w = lane < kEmitThreads / 32 ? s_warp[lane] : 0;
        const int32_t incl = warp_incl_scan(w);
        const int32_t total = __shfl_sync(FULL, incl, 31);
        if (lane < kEmitThreads / 32) s_warp[lane] = incl - w;
        const int64_t excl = lookback(f.emit_states, lt, total, status);
        if (lane == 0) {
            s_excl = excl;
            if (lt == ntiles - 1) {
                *f.ngroups = excl + total;
                if (excl + total > f.max_groups) set_status(status, PX_ERR_CAPACITY);
            }
        }
    }
    __syncthreads();
    // Every item's value of an aggregate is loaded before any is stored: the stores
    // would otherwise hold back the next loads, one memory round trip per item (22
    // tiles of six fragments: 15.8 us for this kernel).
    const uint32_t ltm = lanemask_lt();
    int64_t q[kEmitItems];  // output row, or -1
    int64_t pos = s_excl + s_warp[warp];
#pragma unroll
    for (int i = 0; i < kEmitItems; ++i) {
        q[i] = pos + __popc(mask[i] & ltm);
        if (!((mask[i] >> lane) & 1u) || q[i] >= f.max_groups) q[i] = -1;
        pos += __popc(mask[i]);
        if (q[i] >= 0) store_int(f.out_keys, f.group_w, q[i], f.group_lo + base + i * 32 + lane);
    }
    for (int a = 0; a < f.naggs; ++a) {
        const unsigned long long* acc = f.acc + a * D + base + lane;
        int64_t* out = f.out_aggs[a];
        unsigned long long v[kEmitItems];
#pragma unroll
        for (int i = 0; i < kEmitItems; ++i)
            if (q[i] >= 0) v[i] = acc[i * 32];
#pragma unroll
        for (int i = 0; i < kEmitItems; ++i)
            if (q[i] >= 0) out[q[i]] = static_cast<int64_t>(v[i]);
    }
}

bool valid_type(int32_t t) { return t == PX_I8 || t == PX_I32 || t == PX_I64; }

struct WsLayout {
    size_t plan, counters, acc, states, total;
};

// Accumulator bytes of fragment f: naggs x D 64-bit words, then D occupancy flags
// when there is no COUNT (256-byte aligned).
size_t frag_acc_bytes(const px_fragment& f) {
    const uint64_t D = static_cast<uint64_t>(f.group_hi - f.group_lo) + 1;
    bool has_count = false;
    for (int a = 0; a < f.naggs; ++a) has_count |= f.aggs[a].op == PX_COUNT;
    return align_up(8 * static_cast<size_t>(f.naggs) * D + (has_count ? 0 : D), 256);
}
size_t frag_state_bytes(const px_fragment& f) {
    const int64_t D = f.group_hi - f.group_lo + 1;
    return align_up(8 * static_cast<size_t>(cdiv(D, kEmitTile)), 256);
}

WsLayout frag_ws_layout(const px_fragment* frags, int32_t n) {
    WsLayout L;
    L.plan = kWsScratch;
    L.counters = L.plan + align_up(plan_layout(n).total, 256);  // cleared with what follows
    L.acc = L.counters + 256;
    size_t acc = 0, st = 0;
    for (int32_t i = 0; i < n; ++i) {
        acc += frag_acc_bytes(frags[i]);
        st += frag_state_bytes(frags[i]);
    }
    L.states = L.acc + acc;
    L.total = L.states + st;
    return L;
}

px_status check_fragment(const px_fragment& f, int32_t i) {
    if (f.nrows < 0 || f.nrows > INT32_MAX) return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d nrows", i);
    if (f.key.type != PX_I64 || (f.nrows > 0 && (!f.key.data || !aligned16(f.key.data))))
        return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d key must be an aligned PX_I64 column", i);
    if (f.filter.data && (!valid_type(f.filter.type) || !aligned16(f.filter.data)))
        return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d filter column", i);
    if (f.ncols < 0 || f.ncols > PX_FRAG_MAX_COLS || f.naggs < 0 || f.naggs > PX_FRAG_MAX_AGGS)
        return fail(PX_ERR_UNSUPPORTED, "px_fragments_run: fragment %d has %d columns, %d aggregates", i, f.ncols,
                    f.naggs);
    for (int c = 0; c < f.ncols; ++c)
        if (!valid_type(f.cols[c].type) || (f.nrows > 0 && (!f.cols[c].data || !aligned16(f.cols[c].data))))
            return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d column %d", i, c);
    for (int a = 0; a < f.naggs; ++a) {
        const px_agg& g = f.aggs[a];
        if (g.op != PX_COUNT && g.op != PX_SUM && g.op != PX_SUM_MUL)
            return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d aggregate %d op %d", i, a, g.op);
        if (g.op != PX_COUNT && (g.a < 0 || g.a >= f.ncols))
            return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d aggregate %d column a", i, a);
        if (g.op == PX_SUM_MUL && (g.b < 0 || g.b >= f.ncols))
            return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d aggregate %d column b", i, a);
        if (f.max_groups > 0 && !f.d_out_aggs[a])
            return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d null output aggregate %d", i, a);
    }
    if (!f.d_table || !aligned16(f.d_table)) return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d table", i);
    if (f.nbuild < 0 || !valid_type(f.group.type) || (f.nbuild > 0 && !f.group.data))
        return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d group column", i);
    if (f.group_hi < f.group_lo ||
        static_cast<uint64_t>(f.group_hi) - static_cast<uint64_t>(f.group_lo) >= static_cast<uint64_t>(PX_FRAG_MAX_GROUPS))
        return fail(PX_ERR_UNSUPPORTED, "px_fragments_run: fragment %d group range [%lld, %lld]", i,
                    (long long)f.group_lo, (long long)f.group_hi);
    if (f.max_groups < 0 || (f.max_groups > 0 && !f.d_out_keys) || !f.d_ngroups)
        return fail(PX_ERR_INVALID, "px_fragments_run: fragment %d outputs", i);
    return PX_OK;
}

template <int THREADS, int ITEMS, int NA, bool W8>
px_status launch_frag_na(const PlanHeader* ph, const int64_t* item_start, const FragDev* fd,
                         unsigned long long* counter, int32_t* status, size_t smem, int bps, cudaStream_t st) {
    auto kernel = frag_kernel<THREADS, ITEMS, NA, W8>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) !=
        cudaSuccess)
        return check_launch("px_fragments_run attribute");
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, THREADS, smem);
    if (per_sm < 1) return fail(PX_ERR_UNSUPPORTED, "px_fragments_run: configuration does not fit an SM");
    const int blocks = sm_count() * std::min(per_sm, bps);
    kernel<<<blocks, THREADS, smem, st>>>(ph, item_start, fd, counter, status);
    note_launch();
    return check_launch("px_fragments_run fused");
}

// NA: the batch's largest aggregate count (at least 1), a compile-time bound.
template <int THREADS, int ITEMS, bool W8>
px_status launch_frag(int na, const PlanHeader* ph, const int64_t* item_start, const FragDev* fd,
                      unsigned long long* counter, int32_t* status, size_t smem, int bps, cudaStream_t st) {
    switch (na) {
        case 0:
        case 1: return launch_frag_na<THREADS, ITEMS, 1, W8>(ph, item_start, fd, counter, status, smem, bps, st);
        case 2: return launch_frag_na<THREADS, ITEMS, 2, W8>(ph, item_start, fd, counter, status, smem, bps, st);
        case 3: return launch_frag_na<THREADS, ITEMS, 3, W8>(ph, item_start, fd, counter, status, smem, bps, st);
        default: return launch_frag_na<THREADS, ITEMS, 4, W8>(ph, item_start, fd, counter, status, smem, bps, st);
    }
}

}  // namespace
}  // namespace px

using namespace px;

extern "C" {

size_t px_fragments_plan_bytes(int32_t nfrags) { return plan_layout(nfrags < 0 ? 0 : nfrags).total; }

size_t px_fragments_ws_bytes(const px_fragment* frags, int32_t nfrags) {
    if (!frags || nfrags < 0) return kWsScratch + 256;
    return frag_ws_layout(frags, nfrags).total;
}

px_status px_fragments_run(const px_fragment* frags, int32_t nfrags, const px_fragments_config* cfg, void* h_plan,
                           size_t plan_bytes, void* d_ws, size_t ws_bytes, void* stream) {
    CallRange nvtx_range("px_fragments_run");
    set_error("");
    if (nfrags < 0 || (nfrags > 0 && !frags)) return fail(PX_ERR_INVALID, "px_fragments_run: bad fragment list");
    if (nfrags > INT32_MAX / 2) return fail(PX_ERR_UNSUPPORTED, "px_fragments_run: too many fragments");
    for (int32_t i = 0; i < nfrags; ++i) {
        const px_status s = check_fragment(frags[i], i);
        if (s != PX_OK) return s;
    }
    px_fragments_config c = {512, 2, 0, 2};
    if (cfg) c = *cfg;
    if ((c.threads != 256 && c.threads != 512) || (c.items != 2 && c.items != 4) || c.blocks_per_sm < 1 ||
        c.blocks_per_sm > 8 || c.chunk_rows < 0 || c.chunk_rows % (static_cast<int64_t>(c.threads) * c.items) != 0)
        return fail(PX_ERR_INVALID, "px_fragments_run: bad configuration");
    if (c.chunk_rows == 0) {
        // Rows per work item from the batch, in whole tiles of four rows per thread, at most
        // kMaxChunk: about four items per block of the persistent grid; while that would be
        // two tiles or fewer, one item per block (an item costs about 5 us besides its rows:
        // its ticket, plan, clearing and flush; 6 fragments, 724,000 rows: 36 -> 33 us; 64, 2.2M
        // rows: 64 -> 53).
        const int64_t tile = static_cast<int64_t>(c.threads) * kFilterRows;
        int64_t rows = 0;
        for (int32_t i = 0; i < nfrags; ++i) rows += frags[i].nrows;
        int64_t want = cdiv(rows, static_cast<int64_t>(sm_count()) * c.blocks_per_sm);  // a block's rows
        if (want > 8 * tile) want = cdiv(want, 4);
        c.chunk_rows = std::min<int64_t>(std::max<int64_t>(cdiv(want, tile) * tile, tile), cdiv(kMaxChunk, tile) * tile);
    }
    const PlanLayout PL = plan_layout(nfrags);
    if (!h_plan || plan_bytes < PL.total)
        return fail(PX_ERR_INVALID, "px_fragments_run: plan staging of %zu bytes, %zu needed", plan_bytes, PL.total);
    const WsLayout L = frag_ws_layout(frags, nfrags);
    px_status s = check_ws(d_ws, ws_bytes, L.total, "px_fragments_run");
    if (s != PX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (nfrags == 0) return PX_OK;

    // Work order: decreasing fragment size, so the longest fragments start first.
    std::vector<int32_t> order(nfrags);
    for (int32_t i = 0; i < nfrags; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(),
                     [&](int32_t x, int32_t y) { return frags[x].nrows > frags[y].nrows; });

    char* hp = static_cast<char*>(h_plan);
    PlanHeader* ph = reinterpret_cast<PlanHeader*>(hp);
    int64_t* item_start = reinterpret_cast<int64_t*>(hp + PL.items);
    int64_t* emit_start = reinterpret_cast<int64_t*>(hp + PL.emits);
    FragDev* fd = reinterpret_cast<FragDev*>(hp + PL.frags);
    char* ws = static_cast<char*>(d_ws);
    const int64_t tile = static_cast<int64_t>(c.threads) * c.items;
    // Accumulator and emit-state areas are laid out in the caller's order.
    std::vector<size_t> acc_off(nfrags), st_off(nfrags);
    size_t acc = 0, sto = 0;
    for (int32_t i = 0; i < nfrags; ++i) {
        acc_off[i] = acc;
        st_off[i] = sto;
        acc += frag_acc_bytes(frags[i]);
        sto += frag_state_bytes(frags[i]);
    }
    size_t smem = 0;
    bool w8 = true;  // every aggregated column is 8 bytes wide
    int64_t items = 0, emits = 0;
    for (int32_t k = 0; k < nfrags; ++k) {
        const int32_t i = order[k];
        const px_fragment& f = frags[i];
        FragDev& d = fd[k];
        d = FragDev{};
        d.key = static_cast<const int64_t*>(f.key.data);
        d.filter = f.filter.data;
        d.filter_w = f.filter.type;
        d.lo = f.lo;
        d.hi = f.hi;
        d.nrows = f.nrows;
        d.naggs = f.naggs;
        d.count_agg = -1;
        for (int a = 0; a < f.naggs; ++a) {
            const px_agg& g = f.aggs[a];
            d.op[a] = g.op;
            if (g.op != PX_COUNT) {
                d.pa[a] = f.cols[g.a].data;
                d.wa[a] = f.cols[g.a].type;
                w8 = w8 && d.wa[a] == 8;
            }
            d.same[a] = -1;
            for (int e = 0; e < a && g.op != PX_COUNT; ++e)
                if (f.aggs[e].op == PX_SUM && f.aggs[e].a == g.a) d.same[a] = e;
            if (g.op == PX_SUM_MUL) {
                d.pb[a] = f.cols[g.b].data;
                d.wb[a] = f.cols[g.b].type;
                w8 = w8 && d.wb[a] == 8;
            }
            if (g.op == PX_COUNT && d.count_agg < 0) d.count_agg = a;
        }
        if (f.filter.data) {
            d.stream[d.nstream] = f.filter.data;
            d.stream_w[d.nstream++] = f.filter.type;
        }
        d.stream[d.nstream] = f.key.data;
        d.stream_w[d.nstream++] = 8;
        for (int k = 0; k < f.ncols; ++k) {
            bool read = false;
            for (int a = 0; a < f.naggs; ++a)
                read |= (f.aggs[a].op != PX_COUNT && f.aggs[a].a == k) || (f.aggs[a].op == PX_SUM_MUL && f.aggs[a].b == k);
            if (read) {
                d.stream[d.nstream] = f.cols[k].data;
                d.stream_w[d.nstream++] = f.cols[k].type;
            }
        }
        d.t = table_view(const_cast<void*>(f.d_table), 1);
        d.nbuild = f.nbuild;
        d.group = f.group.data;
        d.group_w = f.group.type;
        d.group_lo = f.group_lo;
        d.D = static_cast<uint32_t>(f.group_hi - f.group_lo + 1);
        // Shared mode when the block arrays fit and a work item can be at least 4 D
        // rows (so clearing and flushing them stays a small part of the item).
        const size_t sbytes = 8 * static_cast<size_t>(f.naggs) * d.D + (d.count_agg < 0 ? (d.D + 31) / 32 * 4 : 0);
        const int64_t rows = sbytes <= kSmallAcc ? f.nrows / 4 : std::min<int64_t>(f.nrows, c.chunk_rows) / 8;
        d.shared = sbytes <= kSmemAccBudget && rows >= static_cast<int64_t>(d.D) ? 1 : 0;
        d.chunk = c.chunk_rows;
        if (d.shared) {
            d.chunk = std::max<int64_t>(c.chunk_rows, cdiv(4 * static_cast<int64_t>(d.D), tile) * tile);
            // Replicas of every slot while they stay few enough to clear and flush per
            // item: lanes with the same group then add to different banks.
            while (d.rep_shift < 5 && (static_cast<uint64_t>(d.D) << (d.rep_shift + 1)) <= kRepSlots &&
                   static_cast<int64_t>((static_cast<uint64_t>(d.D) << (d.rep_shift + 1)) * 8) <= d.chunk)
                ++d.rep_shift;
            smem = std::max(smem, (8 * static_cast<size_t>(f.naggs) * d.D << d.rep_shift) +
                                      (d.count_agg < 0 ? (d.D + 31) / 32 * 4 : 0));
        }
        d.acc = reinterpret_cast<unsigned long long*>(ws + L.acc + acc_off[i]);
        d.occ = d.count_agg < 0 ? reinterpret_cast<uint8_t*>(ws + L.acc + acc_off[i]) + 8 * static_cast<size_t>(f.naggs) * d.D
                                : nullptr;
        d.emit_states = reinterpret_cast<uint64_t*>(ws + L.states + st_off[i]);
        d.out_keys = f.d_out_keys;
        for (int a = 0; a < f.naggs; ++a) d.out_aggs[a] = f.d_out_aggs[a];
        d.ngroups = f.d_ngroups;
        d.max_groups = f.max_groups;
        item_start[k] = items;
        emit_start[k] = emits;
        items += cdiv(f.nrows, d.chunk);
        emits += cdiv(static_cast<int64_t>(d.D), kEmitTile);
    }
    item_start[nfrags] = items;
    emit_start[nfrags] = emits;
    *ph = PlanHeader{};
    ph->nfrags = nfrags;
    ph->nitems = items;
    ph->nemit = emits;

    char* dplan = ws + L.plan;
    unsigned long long* counters = reinterpret_cast<unsigned long long*>(ws + L.counters);
    int32_t* status = &static_cast<WsHeader*>(d_ws)->status;
    cudaMemsetAsync(ws + L.counters, 0, L.total - L.counters, st);
    cudaMemcpyAsync(dplan, h_plan, PL.total, cudaMemcpyHostToDevice, st);
    const PlanHeader* d_ph = reinterpret_cast<const PlanHeader*>(dplan);
    const int64_t* d_items = reinterpret_cast<const int64_t*>(dplan + PL.items);
    const int64_t* d_emits = reinterpret_cast<const int64_t*>(dplan + PL.emits);
    const FragDev* d_fd = reinterpret_cast<const FragDev*>(dplan + PL.frags);
    if (items > 0) {
        int na = 0;
        for (int32_t i = 0; i < nfrags; ++i) na = std::max(na, frags[i].naggs);
        const auto go = [&](auto threads, auto per_thread) {
            constexpr int T = decltype(threads)::value, I = decltype(per_thread)::value;
            return w8 ? launch_frag<T, I, true>(na, d_ph, d_items, d_fd, counters, status, smem, c.blocks_per_sm, st)
                      : launch_frag<T, I, false>(na, d_ph, d_items, d_fd, counters, status, smem, c.blocks_per_sm, st);
        };
        const std::integral_constant<int, 256> t256;
        const std::integral_constant<int, 512> t512;
        const std::integral_constant<int, 2> i2;
        const std::integral_constant<int, 4> i4;
        if (c.threads == 256) s = c.items == 2 ? go(t256, i2) : go(t256, i4);
        else s = c.items == 2 ? go(t512, i2) : go(t512, i4);
        if (s != PX_OK) return s;
    }
    // launch_after only behind a kernel: with no rows the work before is the plan's copy
    const dim3 grid(static_cast<unsigned>(emits));
    if (items > 0)
        launch_after(frag_emit_kernel, grid, dim3(kEmitThreads), 0, st, d_ph, d_emits, d_fd, counters + 1, status);
    else
        frag_emit_kernel<<<grid, kEmitThreads, 0, st>>>(d_ph, d_emits, d_fd, counters + 1, status);
    note_launch();
    return check_launch("px_fragments_run emit");
}

}  // extern "C"

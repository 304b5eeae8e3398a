// px_groupby_agg: HashAggregation (Sec. 3.2) in Single mode, or Partial mode per
// segment (partition) when segments are given; a Final merge is another call.
//
// Group key: the key columns (and the segment id) packed into one 64-bit code,
// each key biased by its sign bit so the code orders like the signed tuple.
// Blocks are persistent over contiguous ranges of positions, which they walk segment
// by segment. With a key-range statistic that makes the key space small, a block
// aggregates into dense shared-memory arrays indexed by the key offset, replicated per
// warp when they fit (fewer same-address atomics), and merges them into the global
// result when the segment ends; rows outside the range take the claim table: slots of
// a table in the workspace claimed with a CAS on a state word (empty -> claimed ->
// published), each taking the next output row, accumulated with 64-bit reductions
// straight into the output columns.
// Without such a statistic: groupby_hash_kernel, an open-addressing table of keys and
// accumulators in the workspace with a small block-local cache in front of it, and
// hash_emit_kernel, which writes its groups out. Of a table for many groups only as much is
// used as an estimate says (hash_estimate_kernel); in a stream of calls a group keeps its
// output row, and small calls write out the groups that they touch (hash_emit_marked_kernel).
// Rows of one warp with lane 0's group are first combined across the warp, so a hot
// key costs one update per warp, not 32.
// All arithmetic is mod 2^64. Every thread loads all of its rows' inputs for a
// tile before aggregating any of them, so each thread keeps many loads in flight.
#include <algorithm>
#include <type_traits>

#include "px_common.cuh"
#include "px_table.cuh"

namespace px {
namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 4;
constexpr int kTile = kThreads * kItems;
constexpr int kMajority = 6;  // smallest group worth a warp reduction
constexpr size_t kSmemBudget = 192 * 1024;
// Dense slots with their replicas, at most (unless one replica has more): more cost
// their clearing and flushing per segment (1000 groups in 64 segments, 2M rows: 8
// replicas 59 us, 2 replicas 45).
constexpr uint64_t kRepSlots = 2048;
constexpr int64_t kDirectRows = 256;  // rows per slot up to which few rows go straight to the global array

struct Spec {
    int32_t nkeys, keybits, segbits, nsegs;
    int32_t key_w[PX_MAX_KEYS];
    const void* key_in[PX_MAX_KEYS];
    void* key_out[PX_MAX_KEYS];
    int32_t naggs;
    int32_t op[PX_MAX_AGGS];
    int32_t a_w[PX_MAX_AGGS], b_w[PX_MAX_AGGS];
    const void* a_in[PX_MAX_AGGS];
    const void* b_in[PX_MAX_AGGS];
    int64_t* agg_out[PX_MAX_AGGS];
    // dense mode: per replica, SUM-like aggregates as low words [n64][D] then high words
    // [n64][D], COUNT aggregates as words [n32][D] (a block counts < 2^32 rows per
    // segment), then an occupancy bitmap when there is no COUNT. The replicas of a word
    // sit side by side, so lanes with replicas of their own use banks of their own.
    int32_t dense;      // 1: dense block arrays
    int32_t rep_shift;  // log2 of the replicas (0..5): a lane uses replica lane mod replicas
    int32_t count_agg;  // a COUNT aggregate marks occupancy; -1: use the bitmap
    uint32_t D;         // dense slots per replica
    int32_t n64, n32;
    int32_t kind[PX_MAX_AGGS];  // 0: u64 array, 1: u32 array
    int32_t slot[PX_MAX_AGGS];  // index of the aggregate's array within its kind
    int32_t sum_agg[PX_MAX_AGGS];  // the aggregates that are not COUNT, in slot order
    uint32_t rep_words;         // words per replica
    int64_t lo[PX_MAX_KEYS];
    uint64_t span[PX_MAX_KEYS];
    // dense global result (when the whole (segment, key) space fits max_groups)
    int32_t dglobal;
    int32_t direct;               // rows update the dense global array directly (no block arrays)
    uint64_t E;                   // entries: max(nsegs, 1) * D
    unsigned long long* dg_acc;   // [naggs][E]
    uint8_t* dg_occ;              // [E] occupancy flags, 1 where the entry has rows (only without COUNT)
    // fused probe (px_join_probe_agg): the key of position j is group[build row of
    // fk[j] in segment q of the table], or no group when fk[j] has no match
    const int64_t* probe_fk;
    TableView probe_t;
    const void* group_col;
    int32_t group_w;
    int64_t nbuild;
};

struct GTable {
    uint32_t* state;              // 0 empty, 1 claimed, 2 published
    unsigned long long* key;
    int32_t* gidx;                // output row of the group, -1 past capacity
    unsigned long long* ngroups;  // groups claimed so far
    uint32_t mask;
    uint32_t most;                // groups from which on the table is given up
};

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint64_t bits_mask(int bits) { return bits >= 64 ? ~0ull : ((1ull << bits) - 1); }

// Group code of key values k0 (, k1) (sign-extended) in segment q.
__device__ __forceinline__ uint64_t compose(const Spec& sp, int64_t k0, int64_t k1, int q) {
    const int b0 = 8 * sp.key_w[0];
    uint64_t code = (static_cast<uint64_t>(k0) ^ (1ull << (b0 - 1))) & bits_mask(b0);
    if (sp.nkeys > 1) {
        const int b1 = 8 * sp.key_w[1];
        code = (code << b1) | ((static_cast<uint64_t>(k1) ^ (1ull << (b1 - 1))) & bits_mask(b1));
    }
    if (sp.segbits) code |= static_cast<uint64_t>(q) << sp.keybits;
    return code;
}

__device__ __forceinline__ void write_group(const Spec& sp, uint64_t code, int32_t gi, int32_t* out_seg) {
    int shift = sp.keybits;
    for (int k = 0; k < sp.nkeys; ++k) {
        const int bits = 8 * sp.key_w[k];
        shift -= bits;
        const uint64_t u = (code >> shift) & bits_mask(bits);
        // u = raw ^ sb; sign-extending raw is (raw ^ sb) - sb = u - sb.
        const uint64_t sb = 1ull << (bits - 1);
        store_int(sp.key_out[k], sp.key_w[k], gi, static_cast<int64_t>(u - sb));
    }
    if (out_seg) out_seg[gi] = sp.segbits ? static_cast<int32_t>(code >> sp.keybits) : 0;
}

// A table of more groups than the output holds is given up before it is full: the result
// is over capacity anyway, and every row of an absent group would walk the longer the
// fuller the table is, in the end all of it. 1M distinct keys, capacity 20,000: this table
// 670 ms, now 0.73; hash mode (see kWalk) 34 ms, now 0.52. A table of up to kFilledSlots is filled whole.
constexpr uint32_t kFilledSlots = 16384;

// Output row of a group code, claiming a slot (and a row) on first sight.
__device__ int32_t global_group(const GTable& g, const Spec& sp, uint64_t code, int64_t max_groups, int32_t* out_seg,
                                int32_t* status) {
    uint32_t s = static_cast<uint32_t>(fmix64(code)) & g.mask;
    for (uint32_t probe = 0; probe <= g.mask; ++probe) {
        if (probe % 64 == 8 && *static_cast<volatile unsigned long long*>(g.ngroups) > g.most) break;
        uint32_t st = ld_acquire_u32(&g.state[s]);
        if (st == 0) {
            st = atomicCAS(&g.state[s], 0u, 1u);
            if (st == 0) {
                const unsigned long long idx = atomicAdd(g.ngroups, 1ull);
                const int32_t gi = idx < static_cast<unsigned long long>(max_groups) ? static_cast<int32_t>(idx) : -1;
                g.key[s] = code;
                g.gidx[s] = gi;
                if (gi >= 0) {
                    write_group(sp, code, gi, out_seg);
                    // The row's accumulators start at zero (an output row may hold an
                    // earlier call's value when calls accumulate into one table).
                    for (int a = 0; a < sp.naggs; ++a) sp.agg_out[a][gi] = 0;
                } else {
                    set_status(status, PX_ERR_CAPACITY);
                }
                __threadfence();
                atomicExch(&g.state[s], 2u);
                return gi;
            }
            // The CAS lost to another claimer; it carries no acquire ordering, so
            // read the state again with one before trusting key and gidx.
            st = ld_acquire_u32(&g.state[s]);
        }
        uint32_t spins = 0;
        while (st == 1) {
            if (++spins > kSpinLimit) {
                set_status(status, PX_ERR_TIMEOUT);
                return -1;
            }
            __nanosleep(32);
            st = ld_acquire_u32(&g.state[s]);
        }
        if (g.key[s] == code) return g.gidx[s];
        s = (s + 1) & g.mask;
    }
    set_status(status, PX_ERR_TABLE_FULL);
    return -1;
}

__device__ __forceinline__ void global_add(const GTable& g, const Spec& sp, uint64_t code, const uint64_t* v,
                                           int64_t max_groups, int32_t* out_seg, int32_t* status) {
    const int32_t gi = global_group(g, sp, code, max_groups, out_seg, status);
    if (gi < 0) return;
    for (int a = 0; a < sp.naggs; ++a)
        red_add_global(reinterpret_cast<unsigned long long*>(&sp.agg_out[a][gi]), static_cast<unsigned long long>(v[a]));
}

// The dense block arrays (see Spec): word w of replica r is word[(w << rep_shift) + r].
// Each 64-bit sum is two 32-bit words, so every update is a native 32-bit shared
// atomic: a 64-bit shared atomicAdd retries under contention and collapses on hot keys.
struct Smem {
    uint32_t* word;
    uint32_t lo, hi, u32, occ;  // first words of the low, high, count and occupancy words
    uint32_t occ_words;
};

__device__ __forceinline__ Smem dense_smem(const Spec& sp, unsigned char* smem) {
    Smem m;
    m.word = reinterpret_cast<uint32_t*>(smem);
    m.lo = 0;
    m.hi = sp.n64 * sp.D;
    m.u32 = 2 * m.hi;
    m.occ = m.u32 + sp.n32 * sp.D;
    m.occ_words = (sp.D + 31) / 32;
    return m;
}

// Adds x (mod 2^64) to the 64-bit value held as words lo/hi: the returned old low
// word tells whether the low addition wrapped; the high word changes only when x
// has high bits or the low word carried. Exact once all updates have landed.
__device__ __forceinline__ void add_split_atomic(uint32_t* lo, uint32_t* hi, uint64_t x) {
    const uint32_t xl = static_cast<uint32_t>(x), xh = static_cast<uint32_t>(x >> 32);
    const uint32_t old = atomicAdd(lo, xl);
    const uint32_t add_hi = xh + (old + xl < old ? 1u : 0u);
    if (add_hi) red_add_shared(hi, add_hi);
}

__device__ __forceinline__ void clear_block_table(const Spec& sp, const Smem& m) {
    const uint32_t nw = sp.rep_words << sp.rep_shift;
    for (uint32_t i = threadIdx.x; i < nw; i += kThreads) m.word[i] = 0;
}

// Merge the block table (segment q) into the global table and clear it.
__device__ void flush_block_table(const Spec& sp, const Smem& m, int q, const GTable& g, int64_t max_groups,
                                  int32_t* out_seg, int32_t* status) {
    __syncthreads();
    // A warp per slot (lanes over the replicas, then a warp sum) when there are few
    // slots for many replicas: a thread per slot would walk every replica alone
    // while the rest of the block waits at the barrier. With many slots the thread
    // per slot keeps every thread busy and wins (a warp sum costs ~12 thread-slot
    // steps).
    const uint32_t sh = sp.rep_shift, reps = 1u << sh;
    const bool warp_flush = (sp.D + kWarps - 1) / kWarps * 12 < (sp.D + kThreads - 1) / kThreads * reps;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Adds replica r of slot d to v (and occ), and clears it.
    const auto take = [&](uint32_t d, uint32_t r, uint64_t* v, bool* occ) {
        for (int a = 0; a < sp.naggs; ++a) {
            const uint32_t o = sp.slot[a] * sp.D + d;
            if (sp.kind[a] == 0) {
                uint32_t* lo = &m.word[((m.lo + o) << sh) + r];
                uint32_t* hi = &m.word[((m.hi + o) << sh) + r];
                v[a] += (static_cast<uint64_t>(*hi) << 32) | *lo;
                *lo = *hi = 0;
            } else {
                uint32_t* c = &m.word[((m.u32 + o) << sh) + r];
                v[a] += *c;
                *c = 0;
            }
        }
        if (sp.count_agg < 0) *occ |= ((m.word[((m.occ + d / 32) << sh) + r] >> (d % 32)) & 1u) != 0;
    };
    const auto put = [&](uint32_t d, const uint64_t* v) {
        if (sp.dglobal) {
            // Dense global array: entry (segment q, slot d); no hashing, no claim.
            const uint64_t e = static_cast<uint64_t>(q) * sp.D + d;
            for (int a = 0; a < sp.naggs; ++a)
                red_add_global(&sp.dg_acc[a * sp.E + e], static_cast<unsigned long long>(v[a]));
            if (sp.count_agg < 0) sp.dg_occ[e] = 1;  // every writer stores the same value
            return;
        }
        const int64_t k0 = sp.lo[0] + static_cast<int64_t>(d / sp.span[1]);
        const int64_t k1 = sp.nkeys > 1 ? sp.lo[1] + static_cast<int64_t>(d % sp.span[1]) : 0;
        global_add(g, sp, compose(sp, k0, k1, q), v, max_groups, out_seg, status);
    };
    for (uint32_t d = warp_flush ? warp : threadIdx.x; d < sp.D; d += warp_flush ? kWarps : kThreads) {
        uint64_t v[PX_MAX_AGGS];
        bool occ = false;
        for (int a = 0; a < sp.naggs; ++a) v[a] = 0;
        if (warp_flush) {
            for (uint32_t r = lane; r < reps; r += 32) take(d, r, v, &occ);
            for (int a = 0; a < sp.naggs; ++a) v[a] = warp_sum(v[a]);
            occ = __any_sync(FULL, occ);
        } else {  // each thread starts at another replica: another bank
            for (uint32_t r = 0; r < reps; ++r) take(d, (r + lane) & (reps - 1), v, &occ);
        }
        if (sp.count_agg >= 0) occ = v[sp.count_agg] != 0;
        if (occ && (!warp_flush || lane == 0)) put(d, v);
    }
    __syncthreads();
    if (sp.count_agg < 0)
        for (uint32_t i = threadIdx.x; i < m.occ_words << sh; i += kThreads) m.word[(m.occ << sh) + i] = 0;
    __syncthreads();
}

constexpr uint32_t kIdxNone = 0xffffffffu;   // no row at this item
constexpr uint32_t kIdxOutside = 0xfffffffeu;  // key outside the dense range

// v[i] = column value at row[i] (sign-extended), 0 where row[i] < 0. One type
// switch per column, then ITEMS independent loads.
template <typename T, int ITEMS>
__device__ __forceinline__ void load_col_t(const void* p, const int32_t (&row)[ITEMS], int64_t* v) {
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) v[i] = row[i] >= 0 ? static_cast<int64_t>(static_cast<const T*>(p)[row[i]]) : 0;
}
template <int ITEMS>
__device__ __forceinline__ void load_col(const void* p, int w, const int32_t (&row)[ITEMS], int64_t* v) {
    if (w == 8) load_col_t<int64_t>(p, row, v);
    else if (w == 4) load_col_t<int32_t>(p, row, v);
    else load_col_t<int8_t>(p, row, v);
}

// The distinct input columns of the kernels that read rows in runs.
constexpr int kMaxStream = PX_MAX_KEYS + 6;
struct Streams {
    int32_t n;
    int32_t w[kMaxStream];
    const void* col[kMaxStream];
};

Streams input_streams(const Spec& sp) {
    Streams t = {};
    const auto add = [&](const void* p, int32_t w) {
        for (int c = 0; c < t.n; ++c)
            if (t.col[c] == p) return;
        if (!p || t.n == kMaxStream) return;
        t.col[t.n] = p;
        t.w[t.n++] = w;
    };
    for (int k = 0; k < sp.nkeys; ++k) add(sp.key_in[k], sp.key_w[k]);
    for (int a = 0; a < sp.naggs; ++a) {
        add(sp.a_in[a], sp.a_w[a]);
        add(sp.b_in[a], sp.b_w[a]);
    }
    return t;
}

// Starts rows [r0, r1) of every input column on their way to L2: thread c takes column
// c. Columns are 16-byte aligned; the ends are rounded down to 16 bytes. The next
// tile's rows, asked for while this one is aggregated: 60M rows of SUM + COUNT 188 ->
// 178 us, 30M rows of two int8 keys and four aggregates 190 -> 177.
__device__ __forceinline__ void prefetch_rows(const Streams& t, int64_t r0, int64_t r1) {
    const int c = threadIdx.x;
    if (c >= t.n || r0 >= r1) return;
    const int64_t b0 = r0 * t.w[c] & ~int64_t(15), b1 = r1 * t.w[c] & ~int64_t(15);
    if (b1 > b0) prefetch_l2(static_cast<const char*>(t.col[c]) + b0, static_cast<uint32_t>(b1 - b0));
}

// v[i] = column value at row r0 + i, 0 from row ncap on; r0 is a multiple of kItems and
// the column 16-byte aligned, so a full run is one load of 4 to 16 bytes (two of 16 for
// 8-byte columns).
template <typename T>
__device__ __forceinline__ void load_run_t(const void* p, int64_t r0, int64_t ncap, int64_t* v) {
    const T* c = static_cast<const T*>(p) + r0;
    if (r0 + kItems <= ncap) {
        __align__(16) T x[kItems];
        if (sizeof(T) == 8) {
            reinterpret_cast<longlong2*>(x)[0] = reinterpret_cast<const longlong2*>(c)[0];
            reinterpret_cast<longlong2*>(x)[sizeof(T) / 8] = reinterpret_cast<const longlong2*>(c)[sizeof(T) / 8];
        } else if (sizeof(T) == 4) {
            *reinterpret_cast<int4*>(x) = *reinterpret_cast<const int4*>(c);
        } else {
            *reinterpret_cast<int32_t*>(x) = *reinterpret_cast<const int32_t*>(c);
        }
#pragma unroll
        for (int i = 0; i < kItems; ++i) v[i] = static_cast<int64_t>(x[i]);
    } else {
#pragma unroll
        for (int i = 0; i < kItems; ++i) v[i] = r0 + i < ncap ? static_cast<int64_t>(c[i]) : 0;
    }
}
__device__ __forceinline__ void load_run(const void* p, int w, int64_t r0, int64_t ncap, int64_t* v) {
    if (w == 8) load_run_t<int64_t>(p, r0, ncap, v);
    else if (w == 4) load_run_t<int32_t>(p, r0, ncap, v);
    else load_run_t<int8_t>(p, r0, ncap, v);
}

// Dense-mode aggregation of positions [a0, a1) of segment q: keys become slot
// indices at load time, each aggregate is applied with one atomic per row, rows outside the key range take
// the global path afterwards.
// DIRECT: no block arrays; every in-range row (or warp-combined hot key) adds
// straight into the dense global array with 64-bit global reductions. Chosen for
// inputs with few rows per entry, where block arrays would cost more to clear
// and flush than they save (a Final merge of Partial results, say).
// PROBE: the key of each position comes from the fused join probe (see Spec).
template <int NA, bool DIRECT, bool PROBE>
__device__ void aggregate_range_dense(const Spec& sp, const Smem& m, const int32_t* __restrict__ sel, int64_t a0,
                                      int64_t a1, int q, const GTable& g, int64_t max_groups, int32_t* out_seg,
                                      int32_t* status) {
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t sh = sp.rep_shift;
    const bool lane_rep = !DIRECT && sh >= 5;  // every lane of a warp has a replica of its own
    uint32_t* const mine = DIRECT ? nullptr : m.word + (tid & ((1u << sh) - 1));
    uint32_t* const LO = mine + (DIRECT ? 0 : m.lo << sh);
    uint32_t* const HI = mine + (DIRECT ? 0 : m.hi << sh);
    uint32_t* const A32 = mine + (DIRECT ? 0 : m.u32 << sh);
    uint32_t* const OCC = mine + (DIRECT ? 0 : m.occ << sh);
    const uint64_t ebase = static_cast<uint64_t>(q) * sp.D;
    SegGeom geo = {};
    bool group_in_table = false;  // PROBE: the table holds the group column beside the keys
    if (PROBE) {
        geo = seg_geom(sp.probe_t, q);
        group_in_table = sp.probe_t.hdr->pay_src == sp.group_col && sp.probe_t.hdr->pay_w == sp.group_w;
    }
    for (int64_t tb = a0; tb < a1; tb += kTile) {
        int32_t row[kItems];
        uint32_t idx[kItems];
        int64_t pkey[kItems];  // PROBE: the gathered group key
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const int64_t j = tb + i * kThreads + tid;
            row[i] = j < a1 ? (sel ? sel[j] : static_cast<int32_t>(j)) : -1;
        }
        if (PROBE) {
            // Join probe of every position: its key's home bucket (one sector: keys,
            // rows and copied payload values), a walk on in the rare case that bucket
            // is full without it, then the group key: the copied payload value when the
            // table holds the group column, else gathered from the build column.
            int64_t fkv[kItems];
            BucketRegs bv[kItems];
#pragma unroll
            for (int i = 0; i < kItems; ++i) fkv[i] = row[i] >= 0 ? sp.probe_fk[row[i]] : kEmpty;
            const Bucket* const segb = sp.probe_t.bk + geo.b0;
            uint32_t hb[kItems];
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                hb[i] = home_bucket(static_cast<uint64_t>(fkv[i]), geo.nb);
                bv[i] = load_bucket(segb + hb[i]);  // hb < nb: inside the segment
            }
            int32_t brow[kItems], bpay[kItems];
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                brow[i] = -1;
                bpay[i] = 0;
                if (fkv[i] == kEmpty) continue;
                bool end;
                int l = bucket_find(bv[i], fkv[i], &end);
                if (l < 0 && !end) l = walk_find(segb, geo.nb, hb[i], fkv[i], &bv[i]);
                if (l >= 0) {
                    brow[i] = bucket_row(bv[i], l);
                    bpay[i] = bucket_pay(bv[i], l);
                }
            }
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                pkey[i] = brow[i] < 0 ? 0
                                      : (group_in_table ? static_cast<int64_t>(bpay[i])
                                                           : load_int(sp.group_col, sp.group_w, brow[i]));
                const uint64_t o0 = static_cast<uint64_t>(pkey[i] - sp.lo[0]);
                idx[i] = brow[i] < 0 ? kIdxNone : (o0 < sp.span[0] ? static_cast<uint32_t>(o0) : kIdxOutside);
            }
        } else {
            int64_t k0[kItems], k1[kItems];
            load_col(sp.key_in[0], sp.key_w[0], row, k0);
            if (sp.nkeys > 1) load_col(sp.key_in[1], sp.key_w[1], row, k1);
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                pkey[i] = 0;
                const uint64_t o0 = static_cast<uint64_t>(k0[i] - sp.lo[0]);
                const uint64_t o1 = sp.nkeys > 1 ? static_cast<uint64_t>(k1[i] - sp.lo[1]) : 0;
                idx[i] = row[i] < 0 ? kIdxNone
                                    : ((o0 < sp.span[0] && o1 < sp.span[1]) ? static_cast<uint32_t>(o0 * sp.span[1] + o1)
                                                                            : kIdxOutside);
            }
        }
        int64_t v[NA > 0 ? NA : 1][kItems];
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            if (a >= sp.naggs) break;
            if (sp.op[a] == PX_COUNT) {
#pragma unroll
                for (int i = 0; i < kItems; ++i) v[a][i] = 1;
            } else {
                load_col(sp.a_in[a], sp.a_w[a], row, v[a]);
                if (sp.op[a] == PX_SUM_MUL) {
                    int64_t y[kItems];
                    load_col(sp.b_in[a], sp.b_w[a], row, y);
#pragma unroll
                    for (int i = 0; i < kItems; ++i)
                        v[a][i] = static_cast<int64_t>(static_cast<uint64_t>(v[a][i]) * static_cast<uint64_t>(y[i]));
                }
            }
        }
        // Hot keys, unless every lane has a replica of its own: when lane 0's slot is shared
        // by at least kMajority lanes, those
        // rows are summed across the warp (COUNT is the peer count; 64-bit sums are
        // three 32-bit warp reductions) and lane 0 applies them once (many lanes
        // on one address would serialise the shared-memory atomics).
        uint32_t apply[kItems];
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            apply[i] = idx[i];
            if (lane_rep) continue;
            const uint32_t c0 = __shfl_sync(FULL, idx[i], 0);
            const uint32_t mm = __ballot_sync(FULL, idx[i] == c0);
            if (c0 < kIdxOutside && __popc(mm) >= kMajority) {
                const bool in = (mm >> lane) & 1u;
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    if (a >= sp.naggs) break;
                    // The probe-fed kernel keeps the shuffle butterfly: redux.sync's
                    // longer latency measured slower there.
                    const int64_t x = PROBE ? warp_sum(in ? v[a][i] : int64_t(0))
                                    : sp.op[a] == PX_COUNT
                                          ? static_cast<int64_t>(__popc(mm))
                                          : static_cast<int64_t>(warp_sum_u64(in ? static_cast<uint64_t>(v[a][i]) : 0));
                    if (lane == 0) v[a][i] = x;
                }
                if (in && lane != 0) apply[i] = kIdxNone;
            }
        }
        // Apply in-range rows.
        if (DIRECT) {
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                if (apply[i] >= kIdxOutside) continue;
                const uint64_t e = ebase + apply[i];
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    if (a >= sp.naggs) break;
                    red_add_global(&sp.dg_acc[a * sp.E + e], static_cast<unsigned long long>(v[a][i]));
                }
                if (sp.count_agg < 0) sp.dg_occ[e] = 1;  // every writer stores the same value
            }
        }
        uint32_t at[kItems];  // first word of the slot's replicas
#pragma unroll
        for (int i = 0; i < kItems; ++i) at[i] = apply[i] << sh;
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            if (DIRECT || a >= sp.naggs) break;
            const uint32_t off = (sp.slot[a] * sp.D) << sh;
            if (sp.kind[a] == 0) {
                uint32_t* const lo = LO + off;
                uint32_t* const hi = HI + off;
#pragma unroll
                for (int i = 0; i < kItems; ++i) {
                    if (apply[i] >= kIdxOutside) continue;
                    add_split_atomic(&lo[at[i]], &hi[at[i]], static_cast<uint64_t>(v[a][i]));
                }
            } else {
                uint32_t* const c = A32 + off;
#pragma unroll
                for (int i = 0; i < kItems; ++i) {
                    if (apply[i] >= kIdxOutside) continue;
                    red_add_shared(&c[at[i]], static_cast<uint32_t>(v[a][i]));
                }
            }
        }
        if (!DIRECT && sp.count_agg < 0) {
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                if (apply[i] >= kIdxOutside) continue;
                red_or_shared(&OCC[(apply[i] / 32) << sh], 1u << (apply[i] % 32));
            }
        }
        // Rows outside the key range (rare when the statistic is right): global path.
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            if (idx[i] != kIdxOutside) continue;
            const int64_t r = row[i];
            const int64_t k0 = PROBE ? pkey[i] : load_int(sp.key_in[0], sp.key_w[0], r);
            const int64_t k1 = !PROBE && sp.nkeys > 1 ? load_int(sp.key_in[1], sp.key_w[1], r) : 0;
            uint64_t full[PX_MAX_AGGS];
#pragma unroll
            for (int a = 0; a < NA; ++a) full[a] = static_cast<uint64_t>(v[a][i]);
            global_add(g, sp, compose(sp, k0, k1, q), full, max_groups, out_seg, status);
        }
    }
}

// The block-array mode of the common shapes: no selection, NS sums of columns or
// products and at most one COUNT. Each thread takes kItems consecutive rows of a tile aligned to
// kTile with vector loads (rows outside [a0, a1) masked), so widths are looked at once
// per column and thread instead of once per value. Issue bound (2.3 instructions per
// cycle; the loads' latency next; three sums under two keys spill 128 bytes of the 64
// registers). Measured, 20M rows: two int8 keys, 3 sums and COUNT at
// 30M rows 306 -> 189 us; 1000 groups, SUM + SUM_MUL + COUNT 152 -> 109; 2 sums without
// COUNT, 100 groups 134 -> 104.
template <int NS, int NK>
__device__ __forceinline__ void aggregate_runs(const Spec& sp, const Streams& in, const Smem& m, int64_t ncap, int64_t a0, int64_t a1,
                                               int q, const GTable& g, int64_t max_groups, int32_t* out_seg,
                                               int32_t* status) {
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t sh = sp.rep_shift;
    const bool lane_rep = sh >= 5;  // every lane of a warp has a replica of its own
    uint32_t* const mine = m.word + (tid & ((1u << sh) - 1));
    uint32_t* const cnts = mine + (m.u32 << sh);
    const uint32_t hi_off = m.hi << sh, Dsh = sp.D << sh;
    for (int64_t tb = a0 / kTile * kTile; tb < a1; tb += kTile) {
        prefetch_rows(in, tb + kTile, tb + 2 * kTile < a1 ? tb + 2 * kTile : a1);
        const int64_t r0 = tb + static_cast<int64_t>(tid) * kItems;
        // the tile's rows in [a0, a1): first .. first + rows
        const uint32_t first = a0 > tb ? static_cast<uint32_t>(a0 - tb) : 0;
        const uint32_t rows = (a1 - tb < kTile ? static_cast<uint32_t>(a1 - tb) : kTile) - first;
        int64_t k0[kItems], k1[kItems], x[NS][kItems];
        load_run(sp.key_in[0], sp.key_w[0], r0, ncap, k0);
        if (NK > 1) load_run(sp.key_in[1], sp.key_w[1], r0, ncap, k1);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int a = sp.sum_agg[s];
            load_run(sp.a_in[a], sp.a_w[a], r0, ncap, x[s]);
            if (sp.op[a] == PX_SUM_MUL) {
                int64_t y[kItems];
                load_run(sp.b_in[a], sp.b_w[a], r0, ncap, y);
#pragma unroll
                for (int i = 0; i < kItems; ++i)
                    x[s][i] = static_cast<int64_t>(static_cast<uint64_t>(x[s][i]) * static_cast<uint64_t>(y[i]));
            }
        }
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const uint64_t o0 = static_cast<uint64_t>(k0[i] - sp.lo[0]);
            uint32_t d = static_cast<uint32_t>(o0);
            bool inside = o0 < sp.span[0];
            if (NK > 1) {
                const uint64_t o1 = static_cast<uint64_t>(k1[i] - sp.lo[1]);
                inside = inside && o1 < sp.span[1];
                d = d * static_cast<uint32_t>(sp.span[1]) + static_cast<uint32_t>(o1);
            }
            if (!inside) d = kIdxOutside;
            if (static_cast<uint32_t>(tid * kItems + i) - first >= rows) d = kIdxNone;
            uint32_t cnt = 1;
            if (!lane_rep) {
                // Hot keys: lane 0's slot shared by at least kMajority lanes is summed
                // across the warp and applied once by lane 0.
                const uint32_t c0 = __shfl_sync(FULL, d, 0);
                const uint32_t mm = __ballot_sync(FULL, d == c0);
                if (c0 < kIdxOutside && __popc(mm) >= kMajority) {
                    const bool in = (mm >> lane) & 1u;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const uint64_t t = warp_sum_u64(in ? static_cast<uint64_t>(x[s][i]) : 0);
                        if (lane == 0) x[s][i] = static_cast<int64_t>(t);
                    }
                    if (lane == 0) cnt = __popc(mm);
                    else if (in) d = kIdxNone;
                }
            }
            if (d < kIdxOutside) {
                uint32_t* p = mine + (d << sh);
#pragma unroll
                for (int s = 0; s < NS; ++s) add_split_atomic(p + s * Dsh, p + hi_off + s * Dsh, static_cast<uint64_t>(x[s][i]));
                if (sp.count_agg >= 0) red_add_shared(cnts + (d << sh), cnt);
                else red_or_shared(mine + ((m.occ + d / 32) << sh), 1u << (d % 32));
            } else if (d == kIdxOutside) {
                uint64_t full[PX_MAX_AGGS];
                if (sp.count_agg >= 0) full[sp.count_agg] = 1;
#pragma unroll
                for (int s = 0; s < NS; ++s) full[sp.sum_agg[s]] = static_cast<uint64_t>(x[s][i]);
                global_add(g, sp, compose(sp, k0[i], NK > 1 ? k1[i] : 0, q), full, max_groups, out_seg, status);
            }
        }
    }
}

// ---------------------------------------------------------------- hash mode ----
// The table of groups, in the workspace: buckets of four slots (one 32-byte sector of
// keys), one and a half slots or more per possible group, and one slot more for the code whose
// stored form would read as empty. Keys hold ~code, 0 where empty; a slot's
// accumulators sit together. A key is set once, by a CAS, and nothing else is published
// with it: accumulators start at zero (cleared with the keys before the call), so no
// row ever waits for another. A code takes the first empty slot from its home bucket
// on, so a lookup mostly reads one sector and ends at the first empty slot.
struct HTable {
    unsigned long long* emitted;  // the emit's counter (see hash_emit_kernel), zero between calls
    uint32_t* done;           // blocks of the emit done where rows were lost, zero between calls
    unsigned long long* key;  // [slots + 1], 32-byte aligned
    unsigned long long* acc;  // [slots + 1] << shift
    uint32_t slots;           // a multiple of kBucketSlots
    uint32_t* chosen;         // kLoose: the slots that are used (see hash_estimate_kernel)
    uint32_t* row;            // a stream's: [slots + 1], 1 + the slot's output row, 0 where it has none yet
    uint32_t* touched;        // a stream's: one bit per slot, zero between calls
    int32_t shift;
};

constexpr int kHashThreads = 512;
constexpr int kHashItems = 4;  // rows a thread loads at a time
constexpr int kHashTile = kHashThreads * kHashItems;
constexpr int kHashBlocksPerSm = 2;
constexpr size_t kCacheBudget = 64 * 1024;  // the block-local cache
constexpr int kHashMajority = 12;           // smallest group worth a warp reduction here
constexpr uint32_t kNoSlot = 0xffffffffu;
// How a call uses the table: whole; as far as chosen on the device; a stream's, whose
// groups keep their output rows, all written out or (kMarked) those that the call touches.
constexpr int kWhole = 0, kLoose = 1, kStream = 2, kMarked = 3;
constexpr uint32_t kBucketSlots = 4;
constexpr uint64_t kMinHashSlots = 8192;    // see htable_slots

struct KeyBucket {
    unsigned long long k[kBucketSlots];
};

// The keys of a bucket as L2 holds them (no L1: another SM's insert must not stay hidden
// behind a stale line). A key that reads 0 may have been set since; its CAS tells.
__device__ __forceinline__ KeyBucket load_keys(const HTable& h, uint32_t bucket) {
    KeyBucket b;
    asm volatile("ld.relaxed.gpu.global.v4.u64 {%0, %1, %2, %3}, [%4];"
                 : "=l"(b.k[0]), "=l"(b.k[1]), "=l"(b.k[2]), "=l"(b.k[3])
                 : "l"(h.key + static_cast<size_t>(bucket) * kBucketSlots)
                 : "memory");
    return b;
}

// The slot of `inv` in the bucket whose keys are `b`, set there if the bucket has room;
// kNoSlot if it is full of other keys.
__device__ __forceinline__ uint32_t bucket_slot(const HTable& h, uint32_t bucket, const KeyBucket& b,
                                                unsigned long long inv) {
    uint32_t at = kNoSlot, empty = kBucketSlots;
#pragma unroll
    for (int j = kBucketSlots - 1; j >= 0; --j) {
        if (b.k[j] == inv) at = bucket * kBucketSlots + j;
        if (b.k[j] == 0) empty = j;
    }
    if (at == kNoSlot)
        for (uint32_t j = empty; j < kBucketSlots; ++j) {
            const unsigned long long old = atomicCAS(&h.key[bucket * kBucketSlots + j], 0ull, inv);
            if (old == 0 || old == inv) {
                at = bucket * kBucketSlots + j;
                break;
            }
        }
    return at;
}

// Buckets that a lookup walks past its home bucket. As many groups as the output holds take
// 0.4 of the slots, or two thirds; the longest run of full buckets is 17 at load 0.5 and 55 at
// two thirds (simulated, 2^26 buckets), unless the keys were chosen for it. Beyond that the
// table is mostly too small, and a walk through all of it, by every row of an absent group,
// has no end to speak of. Rows that find no slot are `lost` to the kernel: the emit sees to
// them (hash_lost).
constexpr uint32_t kWalk = 64;

// The slot of `inv` from bucket `bucket` on (its first bucket was full); kNoSlot where
// kWalk buckets are full. Kept small: registers that it needs are taken from the kernel
// (the end of the walk decided here: 100,000 groups 208 -> 300 us).
__device__ __noinline__ uint32_t hash_walk(const HTable& h, uint32_t bucket, unsigned long long inv) {
    const uint32_t buckets = h.slots / kBucketSlots;
#pragma unroll 1
    for (uint32_t round = 0; round < kWalk; ++round) {
        bucket = bucket + 1 == buckets ? 0 : bucket + 1;
        const uint32_t at = bucket_slot(h, bucket, load_keys(h, bucket), inv);
        if (at != kNoSlot) return at;
    }
    return kNoSlot;
}

// Tells the emit that a row found no slot.
constexpr unsigned long long kLostBit = 1ull << 63;  // of *HTable::emitted
__device__ __forceinline__ void note_lost(const HTable& h) {
    if (!(*static_cast<volatile unsigned long long*>(h.emitted) & kLostBit)) atomicOr(h.emitted, kLostBit);
}

// Marks a slot for the emit of a stream's small call.
__device__ __forceinline__ void mark_touched(const HTable& h, uint32_t slot) {
    uint32_t* w = &h.touched[slot / 32];
    const uint32_t bit = 1u << (slot % 32);
    uint32_t now;  // from L2: a line in L1 would not show the marks of this call
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(w) : "memory");
    if (!(now & bit)) atomicOr(w, bit);
}

// Two neighbouring 64-bit words of shared memory, read anew.
__device__ __forceinline__ ulonglong2 ld_shared_pair(const unsigned long long* p) {
    ulonglong2 v;
    asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(smem_u32(p)) : "memory");
    return v;
}

// Takes an empty slot of the cache pair at `c` for `inv` (or finds it set meanwhile);
// kNoSlot if other codes took both.
__device__ __forceinline__ uint32_t cache_claim(unsigned long long* c_key, uint32_t c, unsigned long long inv) {
    for (uint32_t j = c; j < c + 2; ++j) {
        const unsigned long long old = atomicCAS(&c_key[j], 0ull, inv);
        if (old == 0 || old == inv) return j;
    }
    return kNoSlot;
}

// GROUP BY without a usable statistic. Each row's code is hashed once; the high hash
// bits name two slots of a block-local cache in shared memory, taken by whichever
// codes come first (a hot code comes early and then costs shared-memory adds only),
// the low bits a slot of the table in the workspace, where the rows the cache does not
// hold are added with 64-bit reductions. NA: number of aggregates when known at compile
// time (0..4), or PX_MAX_AGGS.
// Bound by the 64-bit reductions' traffic where most rows go to the table (L1 72 %, L2 69 %
// busy), else by the latency of the dependent steps at 1024 threads per SM. Measured,
// whole calls, 10M rows, int64 keys, SUM + SUM_MUL + COUNT (240 MB), capacity a quarter
// above the groups, against block tables of 4096 slots probed 8 deep in front of a claimed
// and published table: 100,000 groups 1476 -> 207 us; 1M groups 1480 -> 330; 100 groups 98 ->
// 97; Zipf(1.1), 100,000 groups (this kernel) 1209 -> 153. A cache slot pair is read with one
// 16-byte load and a bucket with one 32-byte load; single-slot probing took 408 us at
// 100,000 groups.
// MODE: kWhole (for kStream too), kLoose or kMarked.
template <int NA, int MODE>
__global__ void __launch_bounds__(kHashThreads, kHashBlocksPerSm)
groupby_hash_kernel(Spec sp, const int32_t* __restrict__ sel, const int64_t* __restrict__ d_n, int64_t ncap,
                    const int64_t* __restrict__ d_seg, HTable h, uint32_t cache_slots) {
    extern __shared__ __align__(16) unsigned char smem[];
    if (MODE == kLoose) h.slots = *h.chosen;
    const uint32_t C = cache_slots;
    unsigned long long* c_key = reinterpret_cast<unsigned long long*>(smem);  // [C], ~code or 0
    uint32_t* c_lo = reinterpret_cast<uint32_t*>(c_key + C);                  // [naggs][C]
    uint32_t* c_hi = c_lo + static_cast<size_t>(sp.naggs) * C;                // [naggs][C]
    const int tid = threadIdx.x, lane = tid & 31;
    for (uint32_t w = tid; w < C * (2 + 2 * sp.naggs); w += kHashThreads) reinterpret_cast<uint32_t*>(smem)[w] = 0;
    __syncthreads();
    const int64_t n = actual_rows(d_n, ncap);
    const int64_t chunk = cdiv(cdiv(n, gridDim.x), kHashTile) * kHashTile;
    const int64_t cb = static_cast<int64_t>(blockIdx.x) * chunk;
    const int64_t ce = n < cb + chunk ? n : cb + chunk;
    int64_t pos = cb;
    while (pos < ce) {
        int q = 0;
        int64_t qend = ce;
        if (sp.nsegs > 1) {
            q = seg_of(d_seg, sp.nsegs, pos);
            if (q + 1 < sp.nsegs) {
                const int64_t e = d_seg[q + 1];
                if (e > pos && e < ce) qend = e;
            }
        }
        for (int64_t tb = pos; tb < qend; tb += kHashTile) {
            int32_t row[kHashItems];
#pragma unroll
            for (int i = 0; i < kHashItems; ++i) {
                const int64_t j = tb + i * kHashThreads + tid;
                row[i] = j < qend ? (sel ? sel[j] : static_cast<int32_t>(j)) : -1;
            }
            unsigned long long inv[kHashItems];  // ~code
            uint32_t bucket[kHashItems], cslot[kHashItems];  // home bucket; cache slot pair
            {
                int64_t k0[kHashItems], k1[kHashItems];
                load_col(sp.key_in[0], sp.key_w[0], row, k0);
                if (sp.nkeys > 1) load_col(sp.key_in[1], sp.key_w[1], row, k1);
#pragma unroll
                for (int i = 0; i < kHashItems; ++i) {
                    const uint64_t code = compose(sp, k0[i], sp.nkeys > 1 ? k1[i] : 0, q);
                    const uint64_t hash = fmix64(code);
                    inv[i] = ~code;
                    bucket[i] = slot_of(hash, h.slots / kBucketSlots);
                    cslot[i] = static_cast<uint32_t>(hash >> 32) & (C - 2);
                }
            }
            int64_t v[NA > 0 ? NA : 1][kHashItems];
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                if (a >= sp.naggs) break;
                if (sp.op[a] == PX_COUNT) {
#pragma unroll
                    for (int i = 0; i < kHashItems; ++i) v[a][i] = 1;
                } else {
                    load_col(sp.a_in[a], sp.a_w[a], row, v[a]);
                    if (sp.op[a] == PX_SUM_MUL) {
                        int64_t y[kHashItems];
                        load_col(sp.b_in[a], sp.b_w[a], row, y);
#pragma unroll
                        for (int i = 0; i < kHashItems; ++i)
                            v[a][i] = static_cast<int64_t>(static_cast<uint64_t>(v[a][i]) * static_cast<uint64_t>(y[i]));
                    }
                }
            }
            bool lead[kHashItems];  // the lane applies the item
#pragma unroll
            for (int i = 0; i < kHashItems; ++i) {
                lead[i] = row[i] >= 0;
                // Hot keys: lane 0's code shared by >= kHashMajority lanes is summed across
                // the warp and applied once by lane 0.
                const unsigned long long c0 = __shfl_sync(FULL, inv[i], 0);
                const uint32_t mm = __ballot_sync(FULL, lead[i] && inv[i] == c0);
                if ((mm & 1u) && __popc(mm) >= kHashMajority) {
                    const bool in = (mm >> lane) & 1u;
#pragma unroll
                    for (int a = 0; a < NA; ++a) {
                        if (a >= sp.naggs) break;
                        const int64_t x = sp.op[a] == PX_COUNT
                                              ? static_cast<int64_t>(__popc(mm))
                                              : static_cast<int64_t>(warp_sum_u64(in ? static_cast<uint64_t>(v[a][i]) : 0));
                        if (lane == 0) v[a][i] = x;
                    }
                    lead[i] = lead[i] && (!in || lane == 0);
                }
            }
            // One row of a thread at a time (two rows' round trips together: the registers
            // spill, 251 us at 100,000 groups).
#pragma unroll
            for (int i = 0; i < kHashItems; ++i) {
                // The cache: either slot of the pair, or an empty one of the two.
                const ulonglong2 ck = ld_shared_pair(c_key + cslot[i]);
                uint32_t c = kNoSlot;
                bool pend = false;  // for the table
                if (lead[i]) {
                    if (inv[i] != 0) {
                        if (ck.x == inv[i]) c = cslot[i];
                        else if (ck.y == inv[i]) c = cslot[i] + 1;
                        else if (ck.x == 0 || ck.y == 0) c = cache_claim(c_key, cslot[i], inv[i]);
                    }
                    pend = c == kNoSlot;
                }
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    if (a >= sp.naggs) break;
                    uint32_t* lo = c_lo + static_cast<uint32_t>(a) * C;
                    if (sp.op[a] == PX_COUNT) {  // a block counts fewer than 2^32 rows
                        if (c != kNoSlot) red_add_shared(&lo[c], static_cast<uint32_t>(v[a][i]));
                    } else if (c != kNoSlot) {
                        add_split_atomic(&lo[c], c_hi + static_cast<uint32_t>(a) * C + c, static_cast<uint64_t>(v[a][i]));
                    }
                }
                KeyBucket kb;
                if (pend) kb = load_keys(h, bucket[i]);
                if (pend) {
                    uint32_t slot;
                    if (inv[i] == 0) {  // the code that reads as empty has a slot of its own
                        slot = h.slots;
                        h.key[slot] = 1;  // every writer stores the same value
                    } else {
                        slot = bucket_slot(h, bucket[i], kb, inv[i]);
                        if (slot == kNoSlot) slot = hash_walk(h, bucket[i], inv[i]);
                    }
                    if (slot == kNoSlot) {
                        note_lost(h);
                    } else {
                        if (MODE == kMarked) mark_touched(h, slot);
                        unsigned long long* acc = h.acc + (static_cast<size_t>(slot) << h.shift);
#pragma unroll
                        for (int a = 0; a < NA; ++a) {
                            if (a >= sp.naggs) break;
                            red_add_global(acc + a, static_cast<unsigned long long>(v[a][i]));
                        }
                    }
                }
            }
        }
        // The cache into the table, then cleared: a next segment's codes are other codes.
        __syncthreads();
        for (uint32_t c = tid; c < C; c += kHashThreads) {
            const unsigned long long ci = c_key[c];
            if (ci == 0) continue;
            const uint32_t home = slot_of(fmix64(~ci), h.slots / kBucketSlots);
            uint32_t slot = bucket_slot(h, home, load_keys(h, home), ci);
            if (slot == kNoSlot) slot = hash_walk(h, home, ci);
            if (slot == kNoSlot) note_lost(h);
            else if (MODE == kMarked) mark_touched(h, slot);
            for (int a = 0; a < sp.naggs; ++a) {
                const uint32_t o = static_cast<uint32_t>(a) * C + c;
                const uint64_t x = (static_cast<uint64_t>(c_hi[o]) << 32) | c_lo[o];
                if (x && slot != kNoSlot) red_add_global(h.acc + (static_cast<size_t>(slot) << h.shift) + a, x);
                c_lo[o] = c_hi[o] = 0;
            }
            c_key[c] = 0;
        }
        __syncthreads();
        pos = qend;
    }
}

constexpr int kEmitThreads = 256;
constexpr int kEmitItems = 8;
constexpr int kEmitTile = kEmitThreads * kEmitItems;
constexpr int kEmitWarps = kEmitThreads / 32;

// Adds the lost rows of a table of `groups` groups, at slots beyond their walk: buckets
// never empty again, so a code that is not among its first kWalk + 1 buckets has no row in
// the table yet. With all_rows: adds every row, wherever its slot is (to a cleared table).
// For one block, alone.
__device__ void hash_lost(const Spec& sp, const int32_t* sel, int64_t n, const int64_t* d_seg, const HTable& h,
                          bool all_rows, int64_t groups, int64_t max_groups, int32_t* status) {
    __shared__ unsigned long long s_groups;
    if (threadIdx.x == 0) s_groups = static_cast<unsigned long long>(groups);
    __syncthreads();
    volatile unsigned long long* now = &s_groups;
    const uint32_t buckets = h.slots / kBucketSlots, from = all_rows ? 0 : kWalk + 1;
    for (int64_t j = threadIdx.x; j < n && *now <= static_cast<unsigned long long>(max_groups); j += blockDim.x) {
        const int64_t r = sel ? sel[j] : j;
        const int q = sp.nsegs > 1 ? seg_of(d_seg, sp.nsegs, j) : 0;
        const uint64_t code = compose(sp, load_int(sp.key_in[0], sp.key_w[0], r),
                                      sp.nkeys > 1 ? load_int(sp.key_in[1], sp.key_w[1], r) : 0, q);
        const unsigned long long inv = ~code;
        uint32_t b = slot_of(fmix64(code), buckets);
        uint32_t slot = kNoSlot;
        bool walked = true;  // past its walk without a slot: a lost row
        if (inv == 0) {      // has a slot of its own
            if (!all_rows) continue;
            slot = h.slots;
            if (atomicExch(&h.key[slot], 1ull) == 0) atomicAdd(&s_groups, 1ull);
        }
        for (uint32_t round = 0; round < buckets && slot == kNoSlot; ++round, b = b + 1 == buckets ? 0 : b + 1) {
            const KeyBucket kb = load_keys(h, b);
            for (uint32_t k = 0; k < kBucketSlots && slot == kNoSlot; ++k) {
                unsigned long long key = kb.k[k];
                if (key == 0 && round >= from) {
                    key = atomicCAS(&h.key[b * kBucketSlots + k], 0ull, inv);
                    if (key == 0) {
                        atomicAdd(&s_groups, 1ull);
                        key = inv;
                    }
                }
                if (key == inv) {
                    slot = b * kBucketSlots + k;
                    walked = round >= from;
                }
            }
        }
        if (slot == kNoSlot) set_status(status, PX_ERR_CAPACITY);
        if (slot == kNoSlot || !walked) continue;
        unsigned long long* acc = h.acc + (static_cast<size_t>(slot) << h.shift);
        for (int a = 0; a < sp.naggs; ++a) {
            uint64_t x = 1;
            if (sp.op[a] != PX_COUNT) x = static_cast<uint64_t>(load_int(sp.a_in[a], sp.a_w[a], r));
            if (sp.op[a] == PX_SUM_MUL) x *= static_cast<uint64_t>(load_int(sp.b_in[a], sp.b_w[a], r));
            red_add_global(acc + a, x);
        }
    }
    __syncthreads();
}

// Writes out the groups in tile `tile` of the table's slots: those without an output row
// (in a stream, the new ones) from the one that first_row(their number) gives thread 0 on.
template <bool STREAM, typename F>
__device__ __forceinline__ void hash_emit_tile(const Spec& sp, const HTable& h, int64_t tile, int64_t max_groups,
                                               int32_t* out_seg, int32_t* s_warp, int64_t* s_base, F first_row) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nslots = static_cast<int64_t>(h.slots) + 1;
    const int64_t base = tile * kEmitTile + warp * (32 * kEmitItems) + lane;
    unsigned long long key[kEmitItems];
#pragma unroll
    for (int i = 0; i < kEmitItems; ++i) key[i] = base + i * 32 < nslots ? h.key[base + i * 32] : 0;
    uint32_t had[kEmitItems];  // STREAM: the output row from earlier calls, as in HTable::row
    uint32_t mask[kEmitItems];
    int32_t cnt = 0;
#pragma unroll
    for (int i = 0; i < kEmitItems; ++i) {
        had[i] = STREAM && key[i] != 0 ? h.row[base + i * 32] : 0;
        mask[i] = __ballot_sync(FULL, key[i] != 0 && had[i] == 0);
        cnt += __popc(mask[i]);
    }
    if (lane == 0) s_warp[warp] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t total = 0;
        for (int w = 0; w < kEmitWarps; ++w) {
            const int32_t c = s_warp[w];
            s_warp[w] = total;
            total += c;
        }
        *s_base = first_row(total);
    }
    __syncthreads();
    const uint32_t lt = lanemask_lt();
    int64_t p[kEmitItems];  // output row, or -1
    int64_t pos = *s_base + s_warp[warp];
#pragma unroll
    for (int i = 0; i < kEmitItems; ++i) {
        p[i] = pos + __popc(mask[i] & lt);
        if (STREAM && had[i]) p[i] = had[i] - 1;
        if (STREAM && key[i] != 0 && !had[i]) h.row[base + i * 32] = static_cast<uint32_t>(p[i]) + 1;
        if (key[i] == 0 || p[i] >= max_groups) p[i] = -1;
        pos += __popc(mask[i]);
        if (p[i] >= 0 && !had[i]) {
            const uint64_t code = base + i * 32 == nslots - 1 ? ~0ull : ~key[i];
            write_group(sp, code, static_cast<int32_t>(p[i]), out_seg);
        }
    }
    for (int a = 0; a < sp.naggs; ++a) {
        const unsigned long long* acc = h.acc + (static_cast<size_t>(base) << h.shift) + a;
        int64_t* out = sp.agg_out[a];
        unsigned long long v[kEmitItems];
#pragma unroll
        for (int i = 0; i < kEmitItems; ++i)
            if (p[i] >= 0) v[i] = acc[static_cast<size_t>(i) * 32 << h.shift];
#pragma unroll
        for (int i = 0; i < kEmitItems; ++i)
            if (p[i] >= 0) out[p[i]] = static_cast<int64_t>(v[i]);
    }
}

// Clears slots [0, slots] of the table, as thread `i` of `n`.
__device__ void hash_clear(const HTable& h, uint32_t slots, size_t i, size_t n) {
    const size_t keys = static_cast<size_t>(slots) + 1, words = keys << h.shift;
    const ulonglong2 zero = {};
    for (size_t k = i; k < keys / 2; k += n) reinterpret_cast<ulonglong2*>(h.key)[k] = zero;
    for (size_t k = i; k < words / 2; k += n) reinterpret_cast<ulonglong2*>(h.acc)[k] = zero;
    if (i == 0) {  // an odd last word
        h.key[keys - 1] = 0;
        h.acc[words - 1] = 0;
    }
}

// The end of the emit where rows were lost, in the `blocks` blocks that emit. If the groups
// exceed the output, that is the result; else (keys chosen to meet in one place) the last
// block to be done adds the lost rows and writes all groups out anew. Where the slots were
// chosen by an estimate, that was too low: the block makes the table of all `most` slots.
template <bool STREAM>
__device__ __noinline__ void hash_emit_lost(const Spec& sp, const HTable& used, uint32_t most, uint32_t blocks,
                                            int64_t max_groups, int32_t* out_seg, int64_t* d_ngroups, int32_t* status,
                                            const int32_t* sel, const int64_t* d_n, int64_t ncap,
                                            const int64_t* d_seg) {
    HTable h = used;
    __shared__ int32_t s_warp[kEmitWarps];
    __shared__ int64_t s_base;
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();  // with the barrier above: the block's output rows
        s_last = atomicAdd(h.done, 1u) == blocks - 1;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    if (threadIdx.x == 0) *h.done = 0;
    int64_t groups = *static_cast<volatile int64_t*>(d_ngroups);
    if (groups > max_groups) return;
    const bool anew = h.slots < most;
    if (anew) {
        h.slots = most;
        hash_clear(h, most, threadIdx.x, blockDim.x);
        groups = 0;
        __syncthreads();
    }
    hash_lost(sp, sel, actual_rows(d_n, ncap), d_seg, h, anew, groups, max_groups, status);
    int64_t run = STREAM ? groups : 0;
    for (int64_t tile = 0; tile < cdiv(static_cast<int64_t>(h.slots) + 1, kEmitTile); ++tile) {
        hash_emit_tile<STREAM>(sp, h, tile, max_groups, out_seg, s_warp, &s_base, [&](int32_t total) {
            run += total;
            return run - total;
        });
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (STREAM) *h.emitted = static_cast<unsigned long long>(run);
        *d_ngroups = run;
        if (run > max_groups) set_status(status, PX_ERR_CAPACITY);
    }
}

// A block's add to *h.emitted for `total` more groups, as one of `parts`; called by one
// thread. Gives the first of their output rows. The low bits count groups (a stream's stay
// from call to call), the high bits parts, and the highest bit tells of lost rows; the last
// part writes the number of groups and clears the rest.
constexpr int kEmittedBits = 40;
__device__ __forceinline__ int64_t take_rows(const HTable& h, int32_t total, int64_t parts, int64_t max_groups,
                                             bool* s_lost, int64_t* d_ngroups, int32_t* status) {
    const unsigned long long old = atomicAdd(h.emitted, (1ull << kEmittedBits) | static_cast<unsigned long long>(total));
    const int64_t first = static_cast<int64_t>(old & ((1ull << kEmittedBits) - 1));
    *s_lost = (old & kLostBit) != 0;
    if (static_cast<int64_t>((old & ~kLostBit) >> kEmittedBits) == parts - 1) {
        *h.emitted = static_cast<unsigned long long>(first + total);
        *d_ngroups = first + total;
        if (first + total > max_groups) set_status(status, PX_ERR_CAPACITY);
    }
    return first;
}

// Writes the table's groups out, in no particular order. A block per tile, or (kLoose) as
// many as are in flight at a time. MODE: kWhole, kLoose or kStream.
template <int MODE>
__global__ void __launch_bounds__(kEmitThreads, 4)
hash_emit_kernel(const __grid_constant__ Spec sp, const __grid_constant__ HTable h0, int64_t max_groups,
                 int32_t* __restrict__ out_seg, int64_t* d_ngroups, int32_t* status, const int32_t* __restrict__ sel,
                 const int64_t* __restrict__ d_n, int64_t ncap, const int64_t* __restrict__ d_seg) {
    __shared__ int32_t s_warp[kEmitWarps];
    __shared__ int64_t s_base;
    __shared__ bool s_lost;
    wait_prior();  // the table
    HTable h = h0;
    int64_t tiles = gridDim.x;
    if (MODE == kLoose) {
        h.slots = *h.chosen;
        tiles = cdiv(static_cast<int64_t>(h.slots) + 1, kEmitTile);
        if (blockIdx.x >= tiles) return;
    }
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        if (MODE == kLoose) __syncthreads();  // the tile before has read s_warp and s_base
        hash_emit_tile<MODE == kStream>(sp, h, tile, max_groups, out_seg, s_warp, &s_base, [&](int32_t total) {
            return take_rows(h, total, tiles, max_groups, &s_lost, d_ngroups, status);
        });
        if (MODE != kLoose) break;
    }
    if (s_lost)
        hash_emit_lost<MODE == kStream>(sp, h, h0.slots, static_cast<uint32_t>(gridDim.x < tiles ? gridDim.x : tiles),
                                        max_groups, out_seg, d_ngroups, status, sel, d_n, ncap, d_seg);
}

// The emit of a stream's small call: a thread per 32 slots, which writes out those that the
// call touched (10,000 rows a call, capacity 10M, 8M groups: 224 us a call with all groups
// written out, now 52).
__global__ void __launch_bounds__(kEmitThreads)
hash_emit_marked_kernel(const __grid_constant__ Spec sp, const __grid_constant__ HTable h, int64_t max_groups,
                        int32_t* __restrict__ out_seg, int64_t* d_ngroups, int32_t* status,
                        const int32_t* __restrict__ sel, const int64_t* __restrict__ d_n, int64_t ncap,
                        const int64_t* __restrict__ d_seg) {
    __shared__ int32_t s_warp[kEmitWarps];
    __shared__ int64_t s_base;
    __shared__ bool s_lost;
    wait_prior();  // the table
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t w = static_cast<int64_t>(blockIdx.x) * kEmitThreads + tid;
    const uint32_t word = w * 32 <= h.slots ? h.touched[w] : 0;
    int32_t fresh = 0;
    for (uint32_t b = word; b; b &= b - 1) fresh += h.row[w * 32 + __ffs(b) - 1] == 0;
    const int32_t incl = warp_incl_scan(fresh);
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (tid == 0) {
        int32_t total = 0;
        for (int k = 0; k < kEmitWarps; ++k) {
            const int32_t c = s_warp[k];
            s_warp[k] = total;
            total += c;
        }
        s_base = take_rows(h, total, gridDim.x, max_groups, &s_lost, d_ngroups, status);
    }
    __syncthreads();
    int64_t pos = s_base + s_warp[warp] + incl - fresh;
    for (uint32_t b = word; b; b &= b - 1) {
        const int64_t slot = w * 32 + __ffs(b) - 1;
        const uint32_t had = h.row[slot];
        const int64_t p = had ? had - 1 : pos++;
        if (!had) h.row[slot] = static_cast<uint32_t>(p) + 1;
        if (p >= max_groups) continue;
        if (!had) write_group(sp, slot == h.slots ? ~0ull : ~h.key[slot], static_cast<int32_t>(p), out_seg);
        for (int a = 0; a < sp.naggs; ++a)
            sp.agg_out[a][p] = static_cast<int64_t>(h.acc[(static_cast<size_t>(slot) << h.shift) + a]);
    }
    if (word) h.touched[w] = 0;
    if (s_lost)
        hash_emit_lost<true>(sp, h, h.slots, gridDim.x, max_groups, out_seg, d_ngroups, status, sel, d_n, ncap, d_seg);
}

// How many slots the table of a large capacity uses: cleared and scanned whole it may cost
// more than the rows do, and rows spread over more memory than they need go slower. Counts
// distinct codes by HyperLogLog (Flajolet et al., 2007) in one row in eight, in two halves:
// as a sample grows its distinct codes grow ever more slowly, so the whole has at most
// d + 14 (d - h) of them, with d in the sample and h in half of it. A count that is too low
// all the same (see hash_emit_lost) costs time, a block's work on all rows, but no rows.
// 10M rows, 3 aggregates, capacity 10M: 100 groups 312 us, now 118; 100,000 groups 1004, now
// 231; 1M groups 1055, now 730; 4.3M groups 1084 and 1088. The estimate itself takes 13 us
// there, a chain of latencies.
constexpr int kEstThreads = 1024;
constexpr int kEstItems = 4;
constexpr int kEstTile = kEstThreads * kEstItems;
constexpr int kEstRegs = 2048;       // registers of one count: standard error 2.3 %
constexpr int kEstRate = 8;          // one tile in so many is read,
constexpr int64_t kEstAll = 1 << 20; // but every one of fewer rows than this
constexpr size_t kEstBytes = 2 * kEstRegs * 4;
// Slots beside those asked for: up to 14 tiles in a row, 57,344 rows, go unread, and their codes
// may occur nowhere else (6M rows, of one key but for 57,344: 66 ms with room for 8192, now 0.14).
constexpr uint64_t kEstRoom = 1 << 18;

__device__ __forceinline__ float hll_count(float sum, int zero) {
    constexpr float m = kEstRegs;
    const float e = 0.7213f / (1.0f + 1.079f / m) * m * m / sum;
    return e <= 2.5f * m && zero > 0 ? m * logf(m / static_cast<float>(zero)) : e;
}

// regs: 2 x kEstRegs words, zero on entry, in memory of the table's keys; done: a counter of
// blocks, zero on entry.
__global__ void __launch_bounds__(kEstThreads)
hash_estimate_kernel(const __grid_constant__ Spec sp, const int32_t* __restrict__ sel, const int64_t* __restrict__ d_n,
                     int64_t ncap, const int64_t* __restrict__ d_seg, HTable h, uint32_t* regs, uint32_t* done) {
    __shared__ uint32_t s_reg[2 * kEstRegs];
    __shared__ float s_sum[3];  // of 2^-register: either half, both
    __shared__ int s_zero[3];
    __shared__ bool s_last;
    const int tid = threadIdx.x;
    allow_dependents();
    for (int k = tid; k < 2 * kEstRegs; k += kEstThreads) s_reg[k] = 0;
    if (tid < 3) {
        s_sum[tid] = 0;
        s_zero[tid] = 0;
    }
    __syncthreads();
    const int64_t n = actual_rows(d_n, ncap);
    const int rate = n >= kEstAll ? kEstRate : 1;
    const int64_t tiles = cdiv(cdiv(n, kEstTile), rate);
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        // a tile of each eight, not always the same one
        const int64_t first = (t * rate + (rate > 1 ? static_cast<int64_t>(fmix64(t) % kEstRate) : 0)) * kEstTile;
        uint32_t* const reg = s_reg + (t & 1) * kEstRegs;
        int32_t row[kEstItems];
#pragma unroll
        for (int i = 0; i < kEstItems; ++i) {
            const int64_t j = first + i * kEstThreads + tid;
            row[i] = j < n ? (sel ? sel[j] : static_cast<int32_t>(j)) : -1;
        }
        int64_t k0[kEstItems], k1[kEstItems];
        load_col(sp.key_in[0], sp.key_w[0], row, k0);
        if (sp.nkeys > 1) load_col(sp.key_in[1], sp.key_w[1], row, k1);
#pragma unroll
        for (int i = 0; i < kEstItems; ++i) {
            if (row[i] < 0) continue;
            const int q = sp.nsegs > 1 ? seg_of(d_seg, sp.nsegs, first + i * kEstThreads + tid) : 0;
            const uint64_t hash = fmix64(compose(sp, k0[i], sp.nkeys > 1 ? k1[i] : 0, q));
            const uint32_t rank = __clzll(hash << 11 | 1024) + 1;
            uint32_t* r = &reg[hash >> 53];
            if (*static_cast<volatile uint32_t*>(r) < rank) atomicMax(r, rank);
        }
    }
    __syncthreads();
    for (int k = tid; k < 2 * kEstRegs; k += kEstThreads)
        if (s_reg[k]) atomicMax(&regs[k], s_reg[k]);
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    float sum[3] = {};
    int zero[3] = {};
    for (int k = tid; k < kEstRegs; k += kEstThreads) {
        const uint32_t a = *static_cast<volatile uint32_t*>(&regs[k]), b = *static_cast<volatile uint32_t*>(&regs[kEstRegs + k]);
        const uint32_t x[3] = {a, b, a > b ? a : b};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            sum[c] += exp2f(-static_cast<float>(x[c]));
            zero[c] += x[c] == 0;
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float w = warp_sum(sum[c]);
        const int z = warp_sum(zero[c]);
        if (tid % 32 == 0) {
            atomicAdd(&s_sum[c], w);
            atomicAdd(&s_zero[c], z);
        }
    }
    __syncthreads();
    if (tid == 0) {
        *done = 0;
        const float d = hll_count(s_sum[2], s_zero[2]);
        const float half = 0.5f * (hll_count(s_sum[0], s_zero[0]) + hll_count(s_sum[1], s_zero[1]));
        float most = 1.1f * d;
        if (rate > 1) most = d + 14.0f * (fmaxf(d - half, 0.0f) + 0.04f * d);  // with two errors' room
        const uint64_t want = static_cast<uint64_t>(2.5f * most) + kEstRoom;
        *h.chosen = static_cast<uint32_t>(want < h.slots ? want / kBucketSlots * kBucketSlots : h.slots);
    }
}

__global__ void hash_clear_kernel(HTable h) {
    wait_prior();  // the slots chosen
    hash_clear(h, *static_cast<volatile uint32_t*>(h.chosen), static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x,
               static_cast<size_t>(gridDim.x) * blockDim.x);
}

// Dense modes: kDenseBlock (block arrays) and kDenseDirect (rows straight into the
// dense global array). MODE must agree with sp.direct: the modes are separate kernels
// so each gets its own register allocation.
constexpr int kDenseBlock = 1, kDenseDirect = 2;

template <int NA, int MODE, bool PROBE = false>
__global__ void __launch_bounds__(kThreads, 1)
groupby_kernel(Spec sp, const int32_t* __restrict__ sel, const int64_t* __restrict__ d_n, int64_t ncap,
               const int64_t* __restrict__ d_seg, GTable g, int64_t max_groups, int32_t* __restrict__ out_seg,
               int32_t* status) {
    extern __shared__ __align__(16) unsigned char smem[];
    Smem m = {};
    if (MODE == kDenseBlock) {
        m = dense_smem(sp, smem);
        clear_block_table(sp, m);
        __syncthreads();
    }

    if (PROBE) {  // a table this call cannot use: no groups (uniform across the block)
        const TableHeader* h = sp.probe_t.hdr;
        const int S = sp.nsegs > 0 ? sp.nsegs : 1;
        if (h->magic != kMagic || h->nsegs != S || h->unique == 0 || h->nbuild > sp.nbuild) {
            if (blockIdx.x == 0 && threadIdx.x == 0)
                set_status(status, h->magic == kMagic && h->unique == 0 ? PX_ERR_UNSUPPORTED : PX_ERR_INVALID);
            return;
        }
    }
    const int64_t n = actual_rows(d_n, ncap);
    const int64_t chunk = cdiv(cdiv(n, gridDim.x), kTile) * kTile;
    const int64_t cb = static_cast<int64_t>(blockIdx.x) * chunk;
    const int64_t ce = n < cb + chunk ? n : cb + chunk;
    int64_t pos = cb;
    while (pos < ce) {
        int q = 0;
        int64_t qend = ce;
        if (sp.nsegs > 1) {
            q = seg_of(d_seg, sp.nsegs, pos);
            if (q + 1 < sp.nsegs) {
                const int64_t e = d_seg[q + 1];
                if (e > pos && e < ce) qend = e;
            }
        }
        if (MODE == kDenseDirect) {
            aggregate_range_dense<NA, true, PROBE>(sp, m, sel, pos, qend, q, g, max_groups, out_seg, status);
        } else {
            aggregate_range_dense<NA, false, PROBE>(sp, m, sel, pos, qend, q, g, max_groups, out_seg, status);
            flush_block_table(sp, m, q, g, max_groups, out_seg, status);
        }
        pos = qend;
    }
}

// See aggregate_runs.
template <int NS, int NK>
__global__ void __launch_bounds__(kThreads, 1)
groupby_runs_kernel(Spec sp, const __grid_constant__ Streams in, const int64_t* __restrict__ d_n, int64_t ncap, const int64_t* __restrict__ d_seg, GTable g,
                    int64_t max_groups, int32_t* __restrict__ out_seg, int32_t* status) {
    extern __shared__ __align__(16) unsigned char smem[];
    const Smem m = dense_smem(sp, smem);
    clear_block_table(sp, m);
    __syncthreads();
    const int64_t n = actual_rows(d_n, ncap);
    const int64_t chunk = cdiv(cdiv(n, gridDim.x), kTile) * kTile;
    const int64_t cb = static_cast<int64_t>(blockIdx.x) * chunk;
    const int64_t ce = n < cb + chunk ? n : cb + chunk;
    int64_t pos = cb;
    while (pos < ce) {
        int q = 0;
        int64_t qend = ce;
        if (sp.nsegs > 1) {
            q = seg_of(d_seg, sp.nsegs, pos);
            if (q + 1 < sp.nsegs) {
                const int64_t e = d_seg[q + 1];
                if (e > pos && e < ce) qend = e;
            }
        }
        aggregate_runs<NS, NK>(sp, in, m, ncap, pos, qend, q, g, max_groups, out_seg, status);
        flush_block_table(sp, m, q, g, max_groups, out_seg, status);
        pos = qend;
    }
}

// Dense aggregation of the most common Partial shape (a join's output grouped by
// the gathered dimension attribute): one key column KT, SUM of one column VT and
// COUNT, no selection and a dense global result. One shared-memory replica of the
// slots serves every warp of the block (20M rows: 25 groups 70 us, against 88 us for
// groupby_runs_kernel with a replica per lane; 3000 groups 75 and 108). Same contract
// as the block arrays of groupby_kernel with far fewer instructions per row: each thread takes ITEMS consecutive rows with
// 16-byte vector loads, the SUM is held as 32-bit words (an atomic add on the low
// word returns the carry into the high word), COUNT is a plain 32-bit reduction,
// hot keys (lane 0's slot shared by >= kMajority lanes) are summed across the warp
// first, and each segment's slots are flushed into the dense global array.
// Rows whose key lies outside the range take the global hash path.
template <typename KT, typename VT, int ITEMS>
__global__ void __launch_bounds__(kThreads, 1)
groupby_sum_count_kernel(Spec sp, const __grid_constant__ Streams in, int32_t sum_slot, int32_t cnt_slot, const int64_t* __restrict__ d_n, int64_t ncap,
                         const int64_t* __restrict__ d_seg, GTable g, int64_t max_groups, int32_t* __restrict__ out_seg,
                         int32_t* status) {
    constexpr int T = kThreads * ITEMS;
    static_assert(ITEMS * sizeof(KT) % 16 == 0 && ITEMS * sizeof(VT) % 16 == 0, "whole 16-byte loads per thread");
    extern __shared__ __align__(16) uint32_t s_acc[];  // low words [D], high words [D], counts [D]
    const uint32_t D = sp.D;
    uint32_t* s_lo = s_acc;
    uint32_t* s_hi = s_acc + D;
    uint32_t* s_cnt = s_acc + 2 * static_cast<size_t>(D);
    const int tid = threadIdx.x, lane = tid & 31;
    for (uint32_t w = tid; w < 3 * D; w += kThreads) s_acc[w] = 0;
    __syncthreads();
    const KT* __restrict__ key = static_cast<const KT*>(sp.key_in[0]);
    const VT* __restrict__ val = static_cast<const VT*>(sp.a_in[sum_slot]);
    const int64_t lo = sp.lo[0];
    const int64_t n = actual_rows(d_n, ncap);
    // Each block owns a contiguous range of whole tiles and walks it segment by segment.
    const int64_t chunk = cdiv(cdiv(n, gridDim.x), T) * T;
    const int64_t cb = static_cast<int64_t>(blockIdx.x) * chunk;
    const int64_t ce = n < cb + chunk ? n : cb + chunk;
    int64_t pos = cb;
    while (pos < ce) {
        int q = 0;
        int64_t qend = ce;
        if (sp.nsegs > 1) {
            q = seg_of(d_seg, sp.nsegs, pos);
            if (q + 1 < sp.nsegs) {
                const int64_t e = d_seg[q + 1];
                if (e > pos && e < ce) qend = e;
            }
        }
        // Tiles aligned to T, rows outside [pos, qend) masked: a tile that straddles
        // a segment boundary is read once for each side.
        for (int64_t tb = pos / T * T; tb < qend; tb += T) {
            prefetch_rows(in, tb + T, tb + 2 * T < qend ? tb + 2 * T : qend);
            const int64_t r0 = tb + static_cast<int64_t>(tid) * ITEMS;
            KT k[ITEMS];
            VT v[ITEMS];
            if (r0 + ITEMS <= ncap) {
#pragma unroll
                for (int c = 0; c < ITEMS * static_cast<int>(sizeof(KT)) / 16; ++c)
                    reinterpret_cast<int4*>(k)[c] = reinterpret_cast<const int4*>(key + r0)[c];
#pragma unroll
                for (int c = 0; c < ITEMS * static_cast<int>(sizeof(VT)) / 16; ++c)
                    reinterpret_cast<int4*>(v)[c] = reinterpret_cast<const int4*>(val + r0)[c];
            } else {
#pragma unroll
                for (int i = 0; i < ITEMS; ++i) {
                    k[i] = r0 + i < ncap ? key[r0 + i] : KT(0);
                    v[i] = r0 + i < ncap ? val[r0 + i] : VT(0);
                }
            }
            uint32_t idx[ITEMS];
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const int64_t r = r0 + i;
                const uint64_t o = static_cast<uint64_t>(static_cast<int64_t>(k[i]) - lo);
                idx[i] = r < pos || r >= qend ? kIdxNone : (o < D ? static_cast<uint32_t>(o) : kIdxOutside);
            }
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const uint32_t c0 = __shfl_sync(FULL, idx[i], 0);
                const uint32_t mm = __ballot_sync(FULL, idx[i] == c0);
                uint64_t x = static_cast<uint64_t>(static_cast<int64_t>(v[i]));
                uint32_t cnt = 1;
                uint32_t d = idx[i];
                if (c0 < kIdxOutside && __popc(mm) >= kMajority) {  // warp-uniform
                    // Lane 0 (always in the group) applies the group's totals; the
                    // group's other lanes drop out; lanes outside it keep their row.
                    const bool in = (mm >> lane) & 1u;
                    const uint64_t total = warp_sum_u64(in ? x : 0);
                    if (lane == 0) {
                        x = total;
                        cnt = __popc(mm);
                    } else if (in) {
                        d = kIdxNone;
                    }
                }
                if (d < kIdxOutside) {
                    const uint32_t xl = static_cast<uint32_t>(x);
                    const uint32_t old = atomicAdd(&s_lo[d], xl);
                    const uint32_t h = static_cast<uint32_t>(x >> 32) + (old + xl < old ? 1u : 0u);
                    if (h) red_add_shared(&s_hi[d], h);
                    red_add_shared(&s_cnt[d], cnt);
                } else if (d == kIdxOutside) {
                    uint64_t full[2];
                    full[sum_slot] = x;
                    full[cnt_slot] = 1;
                    global_add(g, sp, compose(sp, static_cast<int64_t>(k[i]), 0, q), full, max_groups, out_seg, status);
                }
            }
        }
        // Segment q's slots into the dense global array, then cleared for the next.
        __syncthreads();
        const uint64_t ebase = static_cast<uint64_t>(q) * D;
        for (uint32_t d = tid; d < D; d += kThreads) {
            const uint32_t c = s_cnt[d];
            if (c) {
                red_add_global(&sp.dg_acc[sum_slot * sp.E + ebase + d],
                               (static_cast<unsigned long long>(s_hi[d]) << 32) | s_lo[d]);
                red_add_global(&sp.dg_acc[cnt_slot * sp.E + ebase + d], c);
                s_lo[d] = s_hi[d] = s_cnt[d] = 0;
            }
        }
        __syncthreads();
        pos = qend;
    }
}

template <typename KT, typename VT>
px_status launch_sum_count(const Spec& sp, int32_t sum_slot, int32_t cnt_slot, const int64_t* d_n, int64_t ncap,
                           const int64_t* d_seg, const GTable& g, int64_t max_groups, int32_t* out_seg,
                           int32_t* status, cudaStream_t st) {
    constexpr int ITEMS = 16 / sizeof(KT) > 16 / sizeof(VT) ? 16 / sizeof(KT) : 16 / sizeof(VT);
    auto kernel = groupby_sum_count_kernel<KT, VT, ITEMS>;
    const size_t smem = 12 * static_cast<size_t>(sp.D);
    allow_smem(kernel, smem);
    // A block flushes its D slots at every segment end: give each at least 4 D rows.
    const int64_t grid = std::max<int64_t>(
        1, std::min<int64_t>(cdiv(ncap, std::max<int64_t>(kThreads * ITEMS, 4 * static_cast<int64_t>(sp.D))),
                             sm_count()));
    kernel<<<static_cast<unsigned>(grid), kThreads, smem, st>>>(sp, input_streams(sp), sum_slot, cnt_slot, d_n, ncap,
                                                              d_seg, g, max_groups, out_seg, status);
    note_launch();
    return check_launch("px_groupby_agg sum-count");
}

// px_join_probe_agg's SUM + COUNT shape with the lean kernel's accumulation:
// every position's key is looked up in its segment of the join table (one sector:
// keys, build rows and the group column copied beside them; a walk on for the
// keys displaced past their home bucket), its group's dense slot comes from the
// copied value (else from a gather of the group column), and its amount is added
// to the block's slot as in groupby_sum_count_kernel. The joined rows are never
// written. Two positions per thread (one 16-byte load of their keys).
template <typename VT>
__global__ void __launch_bounds__(kThreads, 1)
groupby_probe_sum_count_kernel(Spec sp, int32_t sum_slot, int32_t cnt_slot, const int64_t* __restrict__ d_n,
                               int64_t ncap, const int64_t* __restrict__ d_seg, GTable g, int64_t max_groups,
                               int32_t* __restrict__ out_seg, int32_t* status) {
    constexpr int ITEMS = 2;
    constexpr int T = kThreads * ITEMS;
    extern __shared__ __align__(16) uint32_t s_acc[];  // low words [D], high words [D], counts [D]
    const uint32_t D = sp.D;
    uint32_t* s_lo = s_acc;
    uint32_t* s_hi = s_acc + D;
    uint32_t* s_cnt = s_acc + 2 * static_cast<size_t>(D);
    const int tid = threadIdx.x, lane = tid & 31;
    for (uint32_t w = tid; w < 3 * D; w += kThreads) s_acc[w] = 0;
    __syncthreads();
    const TableHeader* h = sp.probe_t.hdr;
    const int S = sp.nsegs > 0 ? sp.nsegs : 1;
    if (h->magic != kMagic || h->nsegs != S || h->unique == 0 || h->nbuild > sp.nbuild) {  // unusable table
        if (blockIdx.x == 0 && tid == 0)
            set_status(status, h->magic == kMagic && h->unique == 0 ? PX_ERR_UNSUPPORTED : PX_ERR_INVALID);
        return;
    }
    const bool group_in_table = h->pay_src == sp.group_col && h->pay_w == sp.group_w;
    const int64_t* __restrict__ fk = sp.probe_fk;
    const VT* __restrict__ val = static_cast<const VT*>(sp.a_in[sum_slot]);
    const int64_t lo = sp.lo[0];
    const int64_t n = actual_rows(d_n, ncap);
    const int64_t chunk = cdiv(cdiv(n, gridDim.x), T) * T;
    const int64_t cb = static_cast<int64_t>(blockIdx.x) * chunk;
    const int64_t ce = n < cb + chunk ? n : cb + chunk;
    // The keys and amounts of the next tile to visit are loaded while the current
    // tile's buckets are in flight (one memory round trip per tile, not two).
    auto load_tile = [&](int64_t tb, int64_t* k, VT* v) {
        const int64_t r0 = tb + static_cast<int64_t>(tid) * ITEMS;
        if (r0 + ITEMS <= ncap) {
            const longlong2 k2 = *reinterpret_cast<const longlong2*>(fk + r0);
            k[0] = k2.x;
            k[1] = k2.y;
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) v[i] = val[r0 + i];
        } else {
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                k[i] = r0 + i < ncap ? fk[r0 + i] : kEmpty;
                v[i] = r0 + i < ncap ? val[r0 + i] : VT(0);
            }
        }
    };
    int64_t kn[ITEMS];
    VT vn[ITEMS];
    if (cb < ce) load_tile(cb, kn, vn);
    int64_t pos = cb;
    while (pos < ce) {
        int q = 0;
        int64_t qend = ce;
        if (sp.nsegs > 1) {
            q = seg_of(d_seg, sp.nsegs, pos);
            if (q + 1 < sp.nsegs) {
                const int64_t e = d_seg[q + 1];
                if (e > pos && e < ce) qend = e;
            }
        }
        const SegGeom geo = seg_geom(sp.probe_t, q);
        const Bucket* const segb = sp.probe_t.bk + geo.b0;
        for (int64_t tb = pos / T * T; tb < qend; tb += T) {
            const int64_t r0 = tb + static_cast<int64_t>(tid) * ITEMS;
            int64_t k[ITEMS];
            VT v[ITEMS];
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                k[i] = kn[i];
                v[i] = vn[i];
            }
            bool live[ITEMS];
            uint32_t hb[ITEMS];
            BucketRegs bv[ITEMS];
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const int64_t r = r0 + i;
                live[i] = r >= pos && r < qend && k[i] != kEmpty;
                hb[i] = home_bucket(static_cast<uint64_t>(k[i]), geo.nb);
                bv[i] = load_bucket(segb + hb[i]);  // hb < nb: inside the segment
            }
            // next visit: this segment's next tile, or the tile where the next segment starts
            const int64_t nxt = tb + T < qend ? tb + T : (qend < ce ? qend / T * T : -1);
            if (nxt >= 0) load_tile(nxt, kn, vn);
            uint32_t idx[ITEMS];
            int64_t gk[ITEMS];
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                idx[i] = kIdxNone;
                gk[i] = 0;
                if (!live[i]) continue;
                bool end;
                int l = bucket_find(bv[i], k[i], &end);
                if (l < 0 && !end) l = walk_find(segb, geo.nb, hb[i], k[i], &bv[i]);
                if (l < 0) continue;  // no match: no group
                gk[i] = group_in_table ? static_cast<int64_t>(bucket_pay(bv[i], l))
                                       : load_int(sp.group_col, sp.group_w, bucket_row(bv[i], l));
                const uint64_t o = static_cast<uint64_t>(gk[i] - lo);
                idx[i] = o < D ? static_cast<uint32_t>(o) : kIdxOutside;
            }
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const uint32_t c0 = __shfl_sync(FULL, idx[i], 0);
                const uint32_t mm = __ballot_sync(FULL, idx[i] == c0);
                uint64_t x = static_cast<uint64_t>(static_cast<int64_t>(v[i]));
                uint32_t cnt = 1;
                uint32_t d = idx[i];
                if (c0 < kIdxOutside && __popc(mm) >= kMajority) {  // warp-uniform
                    // Lane 0 (always in the group) applies the group's totals; the
                    // group's other lanes drop out; lanes outside it keep their row.
                    const bool in = (mm >> lane) & 1u;
                    const uint64_t total = warp_sum_u64(in ? x : 0);
                    if (lane == 0) {
                        x = total;
                        cnt = __popc(mm);
                    } else if (in) {
                        d = kIdxNone;
                    }
                }
                if (d < kIdxOutside) {
                    const uint32_t xl = static_cast<uint32_t>(x);
                    const uint32_t old = atomicAdd(&s_lo[d], xl);
                    const uint32_t hi = static_cast<uint32_t>(x >> 32) + (old + xl < old ? 1u : 0u);
                    if (hi) red_add_shared(&s_hi[d], hi);
                    red_add_shared(&s_cnt[d], cnt);
                } else if (d == kIdxOutside) {
                    uint64_t full[2];
                    full[sum_slot] = x;
                    full[cnt_slot] = 1;
                    global_add(g, sp, compose(sp, gk[i], 0, q), full, max_groups, out_seg, status);
                }
            }
        }
        // Segment q's slots into the dense global array, then cleared for the next.
        __syncthreads();
        const uint64_t ebase = static_cast<uint64_t>(q) * D;
        for (uint32_t d = tid; d < D; d += kThreads) {
            const uint32_t c = s_cnt[d];
            if (c) {
                red_add_global(&sp.dg_acc[sum_slot * sp.E + ebase + d],
                               (static_cast<unsigned long long>(s_hi[d]) << 32) | s_lo[d]);
                red_add_global(&sp.dg_acc[cnt_slot * sp.E + ebase + d], c);
                s_lo[d] = s_hi[d] = s_cnt[d] = 0;
            }
        }
        __syncthreads();
        pos = qend;
    }
}

template <typename VT>
px_status launch_probe_sum_count(const Spec& sp, int32_t sum_slot, int32_t cnt_slot, const int64_t* d_n, int64_t ncap,
                                 const int64_t* d_seg, const GTable& g, int64_t max_groups, int32_t* out_seg,
                                 int32_t* status, cudaStream_t st) {
    auto kernel = groupby_probe_sum_count_kernel<VT>;
    const size_t smem = 12 * static_cast<size_t>(sp.D);
    allow_smem(kernel, smem);
    const int64_t grid = std::max<int64_t>(
        1, std::min<int64_t>(cdiv(ncap, std::max<int64_t>(kThreads * 2, 4 * static_cast<int64_t>(sp.D))), sm_count()));
    kernel<<<static_cast<unsigned>(grid), kThreads, smem, st>>>(sp, sum_slot, cnt_slot, d_n, ncap, d_seg, g,
                                                              max_groups, out_seg, status);
    note_launch();
    return check_launch("px_join_probe_agg sum-count");
}

// Writes the occupied entries of the dense global array as output groups, in
// (segment, key) order, after the groups the hash path claimed (rows whose keys
// fell outside the key range). Single pass with a bounded look-back.
__global__ void __launch_bounds__(kEmitThreads)
dense_emit_kernel(Spec sp, const unsigned long long* ngroups_hash, int64_t max_groups,
                  int32_t* __restrict__ out_seg, int64_t* __restrict__ d_ngroups, ScanScratch scan, int32_t* status,
                  int64_t ntiles) {
    __shared__ int64_t s_tile;
    __shared__ int64_t s_excl;
    __shared__ int32_t s_warp[kEmitWarps];
    wait_prior();  // the dense global array and the claimed groups
    const int64_t tile = next_tile(scan.counter, &s_tile);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t base = tile * kEmitTile + warp * (32 * kEmitItems);
    const int64_t E = static_cast<int64_t>(sp.E);
    const int64_t first = static_cast<int64_t>(*ngroups_hash);
    uint32_t mask[kEmitItems];
    int32_t cnt = 0;
#pragma unroll
    for (int i = 0; i < kEmitItems; ++i) {
        const int64_t e = base + i * 32 + lane;
        bool occ = false;
        if (e < E)
            occ = sp.count_agg >= 0 ? sp.dg_acc[sp.count_agg * E + e] != 0 : sp.dg_occ[e] != 0;
        mask[i] = __ballot_sync(FULL, occ);
        cnt += __popc(mask[i]);
    }
    if (lane == 0) s_warp[warp] = cnt;
    __syncthreads();
    if (warp == 0) {
        const int32_t w = lane < kEmitWarps ? s_warp[lane] : 0;
        const int32_t incl = warp_incl_scan(w);
        const int32_t total = __shfl_sync(FULL, incl, 31);
        if (lane < kEmitWarps) s_warp[lane] = incl - w;
        const int64_t excl = lookback(scan.states, tile, total, status);
        if (lane == 0) {
            s_excl = excl;
            if (tile == ntiles - 1) {
                *d_ngroups = first + excl + total;
                if (first + excl + total > max_groups) set_status(status, PX_ERR_CAPACITY);
            }
        }
    }
    __syncthreads();
    // Every item's value of an aggregate is loaded before any is stored: the stores would
    // otherwise hold back the next loads, one memory round trip per item (10,000 entries,
    // two aggregates: 12.5 us, now 7.8).
    const uint32_t lt = lanemask_lt();
    int64_t p[kEmitItems];  // output row, or -1
    int64_t pos = first + s_excl + s_warp[warp];
#pragma unroll
    for (int i = 0; i < kEmitItems; ++i) {
        p[i] = pos + __popc(mask[i] & lt);
        if (!((mask[i] >> lane) & 1u) || p[i] >= max_groups) p[i] = -1;
        pos += __popc(mask[i]);
        if (p[i] >= 0) {
            const uint32_t e = static_cast<uint32_t>(base + i * 32 + lane);  // E <= max_groups < 2^31
            const uint32_t q = e / sp.D, d = e % sp.D;
            const uint32_t span1 = static_cast<uint32_t>(sp.span[1]);
            store_int(sp.key_out[0], sp.key_w[0], p[i], sp.lo[0] + static_cast<int64_t>(d / span1));
            if (sp.nkeys > 1) store_int(sp.key_out[1], sp.key_w[1], p[i], sp.lo[1] + static_cast<int64_t>(d % span1));
            if (out_seg) out_seg[p[i]] = static_cast<int32_t>(q);
        }
    }
    for (int a = 0; a < sp.naggs; ++a) {
        const unsigned long long* acc = sp.dg_acc + a * E + base + lane;
        int64_t* out = sp.agg_out[a];
        unsigned long long v[kEmitItems];
#pragma unroll
        for (int i = 0; i < kEmitItems; ++i)
            if (p[i] >= 0) v[i] = acc[i * 32];
#pragma unroll
        for (int i = 0; i < kEmitItems; ++i)
            if (p[i] >= 0) out[p[i]] = static_cast<int64_t>(v[i]);
    }
}

// Slots of a table of up to max_groups (< 2^31) groups: a power of two, two per group or
// more, but no more than 32-bit slot numbers hold; above 2^30 groups that is still more
// than one.
uint32_t gtable_slots(int64_t max_groups) {
    uint32_t G = 1024;
    while (G < 2 * static_cast<uint64_t>(max_groups) && G < (1u << 31)) G <<= 1;
    return G;
}

// Slots of the hash mode's table: two and a half per group, or one and a half where a slot's
// accumulators take 64 bytes, so that the table needs hardly more memory than the dense
// modes (10M groups: 2.42 GB with a power of two of slots, now 1.19); small tables up to four.
// Less to clear, at a load between those of the powers of two (10M rows: 1M groups 352 us,
// now 308; 100,000 208 and 207; 30,000 200 and 206). Not fewer than kMinHashSlots, so that a
// small capacity that is exceeded still gets a full count of a few thousand groups; as many
// as 32-bit slot numbers hold.
uint32_t htable_slots(int64_t max_groups, int naggs, bool stream) {
    const uint64_t m = static_cast<uint64_t>(max_groups);
    uint64_t s = stream ? m * 145 / 100 : m + m / 2;
    if (naggs <= 4) {
        s = 2 * m + (stream ? m / 4 : m / 2);
        if (m <= 1 << 16) s = std::max<uint64_t>(s, gtable_slots(max_groups));
    }
    return static_cast<uint32_t>(std::min<uint64_t>(align_up(std::max(s, kMinHashSlots), kBucketSlots), 0xfffffff0u));
}

// Slots of the hash mode's block-local cache: keys and split accumulators.
uint32_t cache_slots(int naggs) {
    uint32_t s = 4096;
    while (s * (8 + 8 * static_cast<size_t>(naggs)) > kCacheBudget) s >>= 1;
    return s;
}

// log2 of a table slot's accumulators, rounded up to a power of two.
int acc_shift(int naggs) { return naggs <= 1 ? 0 : (naggs == 2 ? 1 : (naggs <= 4 ? 2 : 3)); }

// The table of the hash mode: the offsets of its parts from the keys on, and its bytes.
struct HTableLayout {
    size_t acc, row, touched, total;
};
HTableLayout htable_layout(uint32_t slots, int naggs, bool stream) {
    const size_t n = static_cast<size_t>(slots) + 1;
    HTableLayout L;
    L.acc = align_up(8 * n, 256);
    L.row = L.acc + align_up(8 * n << acc_shift(naggs), 256);
    L.touched = L.row + (stream ? align_up(4 * n, 256) : 0);
    L.total = L.touched + (stream ? align_up(cdiv(n, 32) * 4, 256) : 0);
    return L;
}
// A table that takes more than this to clear is used as far as an estimate of the groups
// says (with 3 aggregates from a capacity of about 1M on). The estimate and its kernels take
// about as long as clearing and scanning 96 MB (10M rows in 100 groups: capacity 1M, without,
// 117 us; capacity 10M, with it, 118).
constexpr size_t kLooseBytes = 96 << 20;
constexpr uint32_t kMarkedSlots = 1 << 19;  // see groupby_impl
constexpr size_t kEmittedBytes = 256;  // HTable::emitted and done, before the table

int num_sms() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

template <int NA, int MODE, bool PROBE = false>
px_status launch_mode(const Spec& sp, size_t smem, const int32_t* sel, const int64_t* d_n, int64_t ncap,
                      const int64_t* d_seg, const GTable& g, int64_t max_groups, int32_t* out_seg, int32_t* status,
                      cudaStream_t st) {
    auto kernel = groupby_kernel<NA, MODE, PROBE>;
    allow_smem(kernel, smem);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, smem);
    // A dense block flushes its D slots into the global result at every segment end,
    // so each block gets at least 4 D rows: fewer blocks for small inputs, whose
    // flushes would otherwise pile same-address atomics onto the global array.
    const int64_t min_rows =
        MODE == kDenseBlock ? std::max<int64_t>(kTile, 4 * static_cast<int64_t>(sp.D)) : kTile;
    const int64_t grid = std::max<int64_t>(
        1, std::min<int64_t>(cdiv(ncap, min_rows), static_cast<int64_t>(num_sms()) * std::max(1, per_sm)));
    kernel<<<static_cast<unsigned>(grid), kThreads, smem, st>>>(sp, sel, d_n, ncap, d_seg, g, max_groups, out_seg,
                                                                status);
    note_launch();
    return check_launch("px_groupby_agg");
}

// The dense modes (sp.dense), fused with the probe or not.
template <int NA>
px_status launch_dense(const Spec& sp, size_t smem, const int32_t* sel, const int64_t* d_n, int64_t ncap,
                       const int64_t* d_seg, const GTable& g, int64_t max_groups, int32_t* out_seg, int32_t* status,
                       cudaStream_t st) {
    const auto go = [&](auto launch) { return launch(sp, smem, sel, d_n, ncap, d_seg, g, max_groups, out_seg, status, st); };
    if (sp.probe_fk)
        return sp.direct ? go(launch_mode<NA, kDenseDirect, true>) : go(launch_mode<NA, kDenseBlock, true>);
    return sp.direct ? go(launch_mode<NA, kDenseDirect>) : go(launch_mode<NA, kDenseBlock>);
}

// Block-array mode of the shapes groupby_runs_kernel takes.
template <int NS, int NK>
px_status launch_runs(const Spec& sp, size_t smem, const int64_t* d_n, int64_t ncap, const int64_t* d_seg,
                      const GTable& g, int64_t max_groups, int32_t* out_seg, int32_t* status, cudaStream_t st) {
    auto kernel = groupby_runs_kernel<NS, NK>;
    allow_smem(kernel, smem);
    const int64_t min_rows = std::max<int64_t>(kTile, 4 * static_cast<int64_t>(sp.D));  // see launch_mode
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(cdiv(ncap, min_rows), num_sms()));
    kernel<<<static_cast<unsigned>(grid), kThreads, smem, st>>>(sp, input_streams(sp), d_n, ncap, d_seg, g, max_groups,
                                                              out_seg, status);
    note_launch();
    return check_launch("px_groupby_agg runs");
}

template <int NA, int MODE>
px_status launch_hash(const Spec& sp, const int32_t* sel, const int64_t* d_n, int64_t ncap, const int64_t* d_seg,
                      const HTable& h, cudaStream_t st) {
    auto kernel = groupby_hash_kernel<NA, MODE>;
    const uint32_t C = cache_slots(sp.naggs);
    const size_t smem = static_cast<size_t>(C) * (8 + 8 * static_cast<size_t>(sp.naggs));
    allow_smem(kernel, smem);
    const int64_t grid = std::min<int64_t>(cdiv(ncap, kHashTile), static_cast<int64_t>(num_sms()) * kHashBlocksPerSm);
    kernel<<<static_cast<unsigned>(grid), kHashThreads, smem, st>>>(sp, sel, d_n, ncap, d_seg, h, C);
    note_launch();
    return check_launch("px_groupby_agg hash");
}

}  // namespace
}  // namespace px

using namespace px;

extern "C" {

// Workspace, dense modes: [header][group counter][emit scan scratch][claim table's
// states (G slots)][dense global: accumulators (naggs x E of PX_MAX_AGGS x max_groups),
// then E occupancy flags][claim table's keys, rows (G slots)], so one memset clears all
// that a call starts from; hash mode: [header][emit counter][table: keys, accumulators
// (G + 1 slots)].
struct WsLayout {
    size_t counter, emit_scan, state, dg_acc, key, gidx, total;
};

WsLayout ws_layout(int64_t max_groups) {
    if (max_groups < 1) max_groups = 1;
    const size_t G = gtable_slots(max_groups);
    const size_t M = static_cast<size_t>(max_groups);
    WsLayout L;
    L.counter = kWsScratch;
    L.emit_scan = L.counter + 256;
    L.state = L.emit_scan + scan_scratch_bytes(cdiv(static_cast<int64_t>(M), kEmitTile));
    L.dg_acc = L.state + align_up(4 * G, 256);
    L.key = L.dg_acc + align_up((8 * PX_MAX_AGGS + 1) * M, 256);
    L.gidx = L.key + align_up(8 * G, 256);
    L.total = L.gidx + align_up(4 * G, 256);
    for (int naggs : {4, PX_MAX_AGGS})
        for (bool stream : {false, true})
            L.total = std::max(L.total, kWsScratch + kEmittedBytes + 32 +
                                            htable_layout(htable_slots(max_groups, naggs, stream), naggs, stream).total);
    return L;
}

size_t px_groupby_ws_bytes(int64_t nrows, int64_t max_groups) {
    (void)nrows;
    return ws_layout(max_groups).total;
}

// The fused join probe of px_join_probe_agg: the key of a position is the group
// column at the build row its fk matches in the table.
struct ProbeSrc {
    const void* table;
    int32_t fk_col;
    const px_col* group;
    int64_t nbuild;
};

static px_status groupby_impl(const px_batch* in, const int32_t* key_cols, int32_t nkeys, const px_agg* aggs,
                              int32_t naggs, const int32_t* d_sel, const int64_t* d_nsel, const int64_t* d_seg,
                              int32_t nsegs, const px_key_range* range, int64_t max_groups, const px_batch* out,
                              int32_t* d_out_seg, int64_t* d_ngroups, int32_t flags, void* d_ws, size_t ws_bytes,
                              void* stream, const ProbeSrc* probe = nullptr) {
    set_error("");
    if (flags & ~(PX_AGG_ACCUMULATE | PX_AGG_STREAM))
        return fail(PX_ERR_INVALID, "px_groupby_agg_stream: unknown flags 0x%x", flags);
    const bool accumulate = (flags & PX_AGG_ACCUMULATE) != 0;
    const bool streaming = accumulate || (flags & PX_AGG_STREAM) != 0;
    px_status s = check_batch(in, "px_groupby_agg in");
    if (s != PX_OK) return s;
    if (nkeys < 1 || nkeys > PX_MAX_KEYS || !key_cols)
        return fail(PX_ERR_UNSUPPORTED, "px_groupby_agg: nkeys %d outside [1, %d]", nkeys, PX_MAX_KEYS);
    if (naggs < 0 || naggs > PX_MAX_AGGS || (naggs > 0 && !aggs))
        return fail(PX_ERR_UNSUPPORTED, "px_groupby_agg: naggs %d outside [0, %d]", naggs, PX_MAX_AGGS);
    if ((d_sel == nullptr) != (d_nsel == nullptr))
        return fail(PX_ERR_INVALID, "px_groupby_agg: d_sel and d_nsel must be given together");
    if (nsegs < 0 || nsegs > PX_MAX_SEGS)
        return fail(PX_ERR_UNSUPPORTED, "px_groupby_agg: nsegs %d outside [0, %d]", nsegs, PX_MAX_SEGS);
    if ((nsegs > 0) != (d_seg != nullptr))
        return fail(PX_ERR_INVALID, "px_groupby_agg: d_seg must be given exactly when nsegs > 0");
    if (max_groups < 1 || max_groups > INT32_MAX)
        return fail(PX_ERR_INVALID, "px_groupby_agg: max_groups %lld", (long long)max_groups);
    if (!d_ngroups) return fail(PX_ERR_INVALID, "px_groupby_agg: null d_ngroups");
    s = check_batch(out, "px_groupby_agg out");
    if (s != PX_OK) return s;
    if (out->ncols != nkeys + naggs)
        return fail(PX_ERR_INVALID, "px_groupby_agg: out has %d columns, %d expected", out->ncols, nkeys + naggs);
    if (out->nrows < max_groups)
        return fail(PX_ERR_INVALID, "px_groupby_agg: out capacity %lld below max_groups", (long long)out->nrows);
    Spec sp = {};
    sp.nkeys = nkeys;
    sp.keybits = 0;
    for (int k = 0; k < nkeys; ++k) {
        if (!probe && (key_cols[k] < 0 || key_cols[k] >= in->ncols))
            return fail(PX_ERR_INVALID, "px_groupby_agg: key column %d out of range", key_cols[k]);
        const px_col& c = probe ? *probe->group : in->cols[key_cols[k]];
        if (out->cols[k].type != c.type)
            return fail(PX_ERR_INVALID, "px_groupby_agg: out key column %d type differs from input key", k);
        sp.key_w[k] = c.type;
        sp.key_in[k] = c.data;
        sp.key_out[k] = out->cols[k].data;
        sp.keybits += 8 * c.type;
    }
    sp.nsegs = nsegs;
    sp.segbits = 0;
    while (nsegs > 1 && (1ll << sp.segbits) < nsegs) ++sp.segbits;
    if (sp.keybits + sp.segbits > 64)
        return fail(PX_ERR_UNSUPPORTED, "px_groupby_agg: %d key bits + %d segment bits exceed 64", sp.keybits,
                    sp.segbits);
    sp.naggs = naggs;
    sp.count_agg = -1;
    for (int a = 0; a < naggs; ++a) {
        const px_agg& ag = aggs[a];
        if (ag.op != PX_COUNT && ag.op != PX_SUM && ag.op != PX_SUM_MUL)
            return fail(PX_ERR_INVALID, "px_groupby_agg: aggregate %d has unknown op %d", a, ag.op);
        sp.op[a] = ag.op;
        sp.a_w[a] = sp.b_w[a] = 8;
        sp.a_in[a] = sp.b_in[a] = nullptr;
        if (ag.op == PX_COUNT && sp.count_agg < 0) sp.count_agg = a;
        if (ag.op != PX_COUNT) {
            if (ag.a < 0 || ag.a >= in->ncols) return fail(PX_ERR_INVALID, "px_groupby_agg: aggregate %d column a", a);
            sp.a_w[a] = in->cols[ag.a].type;
            sp.a_in[a] = in->cols[ag.a].data;
        }
        if (ag.op == PX_SUM_MUL) {
            if (ag.b < 0 || ag.b >= in->ncols) return fail(PX_ERR_INVALID, "px_groupby_agg: aggregate %d column b", a);
            sp.b_w[a] = in->cols[ag.b].type;
            sp.b_in[a] = in->cols[ag.b].data;
        }
        if (out->cols[nkeys + a].type != PX_I64)
            return fail(PX_ERR_INVALID, "px_groupby_agg: aggregate output column %d must be PX_I64", nkeys + a);
        sp.agg_out[a] = static_cast<int64_t*>(out->cols[nkeys + a].data);
    }
    s = check_ws(d_ws, ws_bytes, px_groupby_ws_bytes(in->nrows, max_groups), "px_groupby_agg");
    if (s != PX_OK) return s;

    // Dense modes when the key statistic makes the key space small enough: rows go
    // straight into a dense global array when every (segment, key) entry fits
    // max_groups and there are too few rows to give each SM a block that amortises
    // clearing and flushing D block slots; else dense block arrays when they fit
    // shared memory; else hashing.
    size_t smem = 0;
    sp.dense = 0;
    sp.direct = 0;
    sp.rep_shift = 0;
    sp.span[0] = sp.span[1] = 1;
    if (range) {
        bool ok = true;
        uint64_t D = 1;
        for (int k = 0; k < nkeys && ok; ++k) {
            if (range->hi[k] < range->lo[k]) {
                ok = false;
                break;
            }
            const uint64_t span = static_cast<uint64_t>(range->hi[k]) - static_cast<uint64_t>(range->lo[k]) + 1;
            if (span == 0 || span > (1ull << 24)) ok = false;
            sp.lo[k] = range->lo[k];
            sp.span[k] = span;
            D *= span;
        }
        if (ok && D <= (1ull << 24)) {
            sp.n64 = sp.n32 = 0;
            for (int a = 0; a < naggs; ++a) {
                sp.kind[a] = sp.op[a] == PX_COUNT ? 1 : 0;
                if (!sp.kind[a]) sp.sum_agg[sp.n64] = a;
                sp.slot[a] = sp.kind[a] ? sp.n32++ : sp.n64++;
            }
            size_t per_rep = static_cast<size_t>(sp.n64) * D * 8 + static_cast<size_t>(sp.n32) * D * 4 +
                             (sp.count_agg < 0 ? (D + 31) / 32 * 4 : 0);
            const uint64_t E = static_cast<uint64_t>(nsegs > 0 ? nsegs : 1) * D;
            // A stream of calls keeps its groups in one place: the choice then depends
            // on the statistic and max_groups only, never on the row count.
            // Few rows, but not so many to a slot that their reductions queue at its address
            // (about 10 ns each: 600,000 rows in 25 groups took 243 us directly).
            const bool few_rows =
                streaming ? per_rep > kSmemBudget
                          : cdiv(in->nrows, std::max<int64_t>(kTile, 4 * static_cast<int64_t>(D))) < num_sms() &&
                                (per_rep > kSmemBudget || in->nrows <= kDirectRows * static_cast<int64_t>(D));
            if (E <= static_cast<uint64_t>(max_groups) && few_rows) {
                sp.dense = 1;
                sp.direct = 1;
                sp.D = static_cast<uint32_t>(D);
            } else if (per_rep > 0 && per_rep <= kSmemBudget) {
                sp.dense = 1;
                sp.D = static_cast<uint32_t>(D);
                // Up to one replica per lane.
                while (sp.rep_shift < 5 && (per_rep << (sp.rep_shift + 1)) <= kSmemBudget &&
                       (D << (sp.rep_shift + 1)) <= kRepSlots)
                    ++sp.rep_shift;
                sp.rep_words = static_cast<uint32_t>(per_rep / 4);
                smem = per_rep << sp.rep_shift;
            }
        }
    }
    if (probe) {
        if (!sp.dense)
            return fail(PX_ERR_UNSUPPORTED,
                        "px_join_probe_agg: needs a group key range small enough for dense aggregation");
        sp.probe_fk = static_cast<const int64_t*>(in->cols[probe->fk_col].data);
        sp.probe_t = table_view(const_cast<void*>(probe->table), nsegs > 0 ? nsegs : 1);
        sp.group_col = probe->group->data;
        sp.group_w = probe->group->type;
        sp.nbuild = probe->nbuild;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t* status = &static_cast<WsHeader*>(d_ws)->status;
    const int64_t ncap = in->nrows;
    if (!sp.dense) {
        // Hash mode. A stream of calls keeps one table, so its size must not depend on a
        // call's rows.
        const uint32_t slots = htable_slots(streaming ? max_groups : std::min(max_groups, ncap), naggs, streaming);
        const HTableLayout T = htable_layout(slots, naggs, streaming);
        char* base = static_cast<char*>(d_ws) + kWsScratch;
        // a bucket is one 32-byte load; the caller's workspace is only 16-byte aligned
        char* keys = reinterpret_cast<char*>(align_up(reinterpret_cast<uintptr_t>(base) + kEmittedBytes, 32));
        HTable h;
        h.emitted = reinterpret_cast<unsigned long long*>(base);
        h.done = reinterpret_cast<uint32_t*>(base + 8);
        h.chosen = reinterpret_cast<uint32_t*>(base + 16);
        h.key = reinterpret_cast<unsigned long long*>(keys);
        h.acc = reinterpret_cast<unsigned long long*>(keys + T.acc);
        h.row = streaming ? reinterpret_cast<uint32_t*>(keys + T.row) : nullptr;
        h.touched = streaming ? reinterpret_cast<uint32_t*>(keys + T.touched) : nullptr;
        h.slots = slots;
        h.shift = acc_shift(naggs);
        // A stream's call of few rows marks the groups that it touches; one of many, or into a
        // small table, writes all groups out (10,000 rows: 281,000 slots 41 us marked, 36 all;
        // 2.8M slots 41 and 63; 1M rows into 22.5M slots 208 and 308).
        const int mode = !streaming ? (T.total > kLooseBytes ? kLoose : kWhole)
                                    : (slots > kMarkedSlots && ncap < static_cast<int64_t>(slots) / 8 ? kMarked : kStream);
        if (!accumulate) cudaMemsetAsync(base, 0, kEmittedBytes + 32 + (mode == kLoose ? kEstBytes : T.total), st);
        const int64_t* d_n = d_sel ? d_nsel : in->d_nrows;
        if (ncap > 0) {
            if (mode == kLoose) {
                const int64_t tiles = cdiv(cdiv(ncap, kEstTile), ncap >= kEstAll ? kEstRate : 1);
                hash_estimate_kernel<<<static_cast<unsigned>(std::min<int64_t>(tiles, num_sms())), kEstThreads, 0, st>>>(
                    sp, d_sel, d_n, ncap, d_seg, h, reinterpret_cast<uint32_t*>(keys), h.done);
                note_launch();
                launch_after(hash_clear_kernel, dim3(num_sms() * 8), dim3(256), 0, st, h);
                note_launch();
            }
            const auto go = [&](auto na) {
                constexpr int NA = decltype(na)::value;
                const auto launch = mode == kLoose ? launch_hash<NA, kLoose>
                                                   : (mode == kMarked ? launch_hash<NA, kMarked> : launch_hash<NA, kWhole>);
                return launch(sp, d_sel, d_n, ncap, d_seg, h, st);
            };
            switch (naggs) {
                case 0: s = go(std::integral_constant<int, 0>{}); break;
                case 1: s = go(std::integral_constant<int, 1>{}); break;
                case 2: s = go(std::integral_constant<int, 2>{}); break;
                case 3: s = go(std::integral_constant<int, 3>{}); break;
                case 4: s = go(std::integral_constant<int, 4>{}); break;
                default: s = go(std::integral_constant<int, PX_MAX_AGGS>{}); break;
            }
            if (s != PX_OK) return s;
        }
        int64_t blocks = cdiv(static_cast<int64_t>(slots) + 1, mode == kMarked ? 32 * kEmitThreads : kEmitTile);
        if (mode == kLoose) blocks = std::min<int64_t>(blocks, num_sms() * 4);
        const auto emit = mode == kLoose    ? hash_emit_kernel<kLoose>
                          : mode == kMarked ? hash_emit_marked_kernel
                          : mode == kStream ? hash_emit_kernel<kStream>
                                            : hash_emit_kernel<kWhole>;
        const dim3 grid(static_cast<unsigned>(blocks));
        if (ncap > 0)  // launch_after only behind a kernel: with no rows the work before is a memset
            launch_after(emit, grid, dim3(kEmitThreads), 0, st, sp, h, max_groups, d_out_seg, d_ngroups, status, d_sel,
                         d_n, ncap, d_seg);
        else
            emit<<<grid, kEmitThreads, 0, st>>>(sp, h, max_groups, d_out_seg, d_ngroups, status, d_sel, d_n, ncap, d_seg);
        note_launch();
        return check_launch("px_groupby_agg hash emit");
    }
    const uint32_t G = gtable_slots(max_groups);
    const WsLayout L = ws_layout(max_groups);
    char* ws = static_cast<char*>(d_ws);
    GTable g;
    g.ngroups = reinterpret_cast<unsigned long long*>(ws + L.counter);
    g.state = reinterpret_cast<uint32_t*>(ws + L.state);
    g.key = reinterpret_cast<unsigned long long*>(ws + L.key);
    g.gidx = reinterpret_cast<int32_t*>(ws + L.gidx);
    g.mask = G - 1;
    // (said here: worked out in the loop of global_group it costs the dense kernels 0.3 %)
    g.most = static_cast<uint32_t>(std::max<int64_t>(max_groups, G <= kFilledSlots ? G - 1 : G - G / 16));
    size_t clear_to = L.state + 4ull * G;  // what a call that starts empty clears
    // Dense global result when the whole (segment, key) space fits max_groups.
    sp.dglobal = 0;
    if (sp.dense) {
        const uint64_t E = static_cast<uint64_t>(nsegs > 0 ? nsegs : 1) * sp.D;
        if (E <= static_cast<uint64_t>(max_groups)) {
            sp.dglobal = 1;
            sp.E = E;
            sp.dg_acc = reinterpret_cast<unsigned long long*>(ws + L.dg_acc);
            sp.dg_occ = reinterpret_cast<uint8_t*>(sp.dg_acc + static_cast<uint64_t>(naggs) * E);
            clear_to = L.dg_acc + 8ull * naggs * E + (sp.count_agg < 0 ? E : 0);
        }
    }
    const size_t clear_from = accumulate ? L.emit_scan : L.counter;
    cudaMemsetAsync(ws + clear_from, 0, (accumulate ? L.state : clear_to) - clear_from, st);
    // The lean kernel of the SUM + COUNT shape (see groupby_sum_count_kernel):
    // one key of 4 or 8 bytes, block arrays of a dense global result, no selection, not
    // fused with a probe.
    int32_t sum_slot = -1, cnt_slot = -1;
    if (naggs == 2)
        for (int a = 0; a < 2; ++a) {
            if (sp.op[a] == PX_COUNT) cnt_slot = a;
            else if (sp.op[a] == PX_SUM && (sp.a_w[a] == 8 || sp.a_w[a] == 4)) sum_slot = a;
        }
    const bool sum_count = ncap > 0 && !probe && sp.dense && !sp.direct && sp.dglobal &&
                           d_sel == nullptr && nkeys == 1 && (sp.key_w[0] == 4 || sp.key_w[0] == 8) &&
                           sum_slot >= 0 && cnt_slot >= 0 && 12 * static_cast<size_t>(sp.D) <= kSmemBudget;
    // The same shape fed by the join probe, with the rows' keys looked up in the table.
    const bool probe_sum_count = ncap > 0 && probe && sp.dense && !sp.direct && sp.dglobal &&
                                 d_sel == nullptr && nkeys == 1 && sum_slot >= 0 && cnt_slot >= 0 &&
                                 12 * static_cast<size_t>(sp.D) <= kSmemBudget;
    if (probe_sum_count) {
        const int64_t* d_n = in->d_nrows;
        s = sp.a_w[sum_slot] == 8
                ? launch_probe_sum_count<int64_t>(sp, sum_slot, cnt_slot, d_n, ncap, d_seg, g, max_groups, d_out_seg,
                                                  status, st)
                : launch_probe_sum_count<int32_t>(sp, sum_slot, cnt_slot, d_n, ncap, d_seg, g, max_groups, d_out_seg,
                                                  status, st);
        if (s != PX_OK) return s;
    } else if (sum_count) {
        const int64_t* d_n = in->d_nrows;
        if (sp.key_w[0] == 4 && sp.a_w[sum_slot] == 8)
            s = launch_sum_count<int32_t, int64_t>(sp, sum_slot, cnt_slot, d_n, ncap, d_seg, g, max_groups, d_out_seg,
                                                   status, st);
        else if (sp.key_w[0] == 4)
            s = launch_sum_count<int32_t, int32_t>(sp, sum_slot, cnt_slot, d_n, ncap, d_seg, g, max_groups, d_out_seg,
                                                   status, st);
        else if (sp.a_w[sum_slot] == 8)
            s = launch_sum_count<int64_t, int64_t>(sp, sum_slot, cnt_slot, d_n, ncap, d_seg, g, max_groups, d_out_seg,
                                                   status, st);
        else
            s = launch_sum_count<int64_t, int32_t>(sp, sum_slot, cnt_slot, d_n, ncap, d_seg, g, max_groups, d_out_seg,
                                                   status, st);
        if (s != PX_OK) return s;
    } else if (ncap > 0) {
        const int64_t* d_n = d_sel ? d_nsel : in->d_nrows;
        const auto runs = [&](auto launch) {
            return launch(sp, smem, d_n, ncap, d_seg, g, max_groups, d_out_seg, status, st);
        };
        const auto go = [&](auto launch) {
            return launch(sp, smem, d_sel, d_n, ncap, d_seg, g, max_groups, d_out_seg, status, st);
        };
        const bool as_runs = !probe && !sp.direct && !d_sel && sp.n32 <= 1 && sp.n64 >= 1 && sp.n64 <= 3;
        if (as_runs && sp.n64 == 1) s = nkeys == 1 ? runs(launch_runs<1, 1>) : runs(launch_runs<1, 2>);
        else if (as_runs && sp.n64 == 2) s = nkeys == 1 ? runs(launch_runs<2, 1>) : runs(launch_runs<2, 2>);
        else if (as_runs) s = nkeys == 1 ? runs(launch_runs<3, 1>) : runs(launch_runs<3, 2>);
        else switch (naggs) {
            case 0: s = go(launch_dense<0>); break;
            case 1: s = go(launch_dense<1>); break;
            case 2: s = go(launch_dense<2>); break;
            case 3: s = go(launch_dense<3>); break;
            case 4: s = go(launch_dense<4>); break;
            default: s = go(launch_dense<PX_MAX_AGGS>); break;
        }
        if (s != PX_OK) return s;
    }
    if (sp.dglobal) {
        const int64_t ntiles = cdiv(static_cast<int64_t>(sp.E), kEmitTile);
        const dim3 grid(static_cast<unsigned>(ntiles));
        if (ncap > 0)  // as above
            launch_after(dense_emit_kernel, grid, dim3(kEmitThreads), 0, st, sp, g.ngroups, max_groups, d_out_seg,
                         d_ngroups, scan_scratch(ws + L.emit_scan), status, ntiles);
        else
            dense_emit_kernel<<<grid, kEmitThreads, 0, st>>>(sp, g.ngroups, max_groups, d_out_seg, d_ngroups,
                                                             scan_scratch(ws + L.emit_scan), status, ntiles);
        note_launch();
        return check_launch("px_groupby_agg emit");
    }
    cudaMemcpyAsync(d_ngroups, g.ngroups, sizeof(int64_t), cudaMemcpyDeviceToDevice, st);
    return check_launch("px_groupby_agg count");
}

px_status px_groupby_agg(const px_batch* in, const int32_t* key_cols, int32_t nkeys, const px_agg* aggs,
                         int32_t naggs, const int32_t* d_sel, const int64_t* d_nsel, const int64_t* d_seg,
                         int32_t nsegs, const px_key_range* range, int64_t max_groups, const px_batch* out,
                         int32_t* d_out_seg, int64_t* d_ngroups, void* d_ws, size_t ws_bytes, void* stream) {
    CallRange nvtx_range("px_groupby_agg");
    return groupby_impl(in, key_cols, nkeys, aggs, naggs, d_sel, d_nsel, d_seg, nsegs, range, max_groups, out,
                        d_out_seg, d_ngroups, 0, d_ws, ws_bytes, stream);
}

px_status px_groupby_agg_stream(const px_batch* in, const int32_t* key_cols, int32_t nkeys, const px_agg* aggs,
                                int32_t naggs, const int32_t* d_sel, const int64_t* d_nsel, const int64_t* d_seg,
                                int32_t nsegs, const px_key_range* range, int64_t max_groups, const px_batch* out,
                                int32_t* d_out_seg, int64_t* d_ngroups, int32_t flags, void* d_ws, size_t ws_bytes,
                                void* stream) {
    CallRange nvtx_range("px_groupby_agg_stream");
    return groupby_impl(in, key_cols, nkeys, aggs, naggs, d_sel, d_nsel, d_seg, nsegs, range, max_groups, out,
                        d_out_seg, d_ngroups, flags, d_ws, ws_bytes, stream);
}

size_t px_join_probe_agg_ws_bytes(int64_t nprobe, int64_t max_groups) { return px_groupby_ws_bytes(nprobe, max_groups); }

px_status px_join_probe_agg(const void* d_table, const px_batch* probe, int32_t fk_col, const int32_t* d_sel,
                            const int64_t* d_nsel, const int64_t* d_seg, int32_t nsegs, const px_col* group,
                            int64_t nbuild, int64_t group_lo, int64_t group_hi, const px_agg* aggs, int32_t naggs,
                            int64_t max_groups, const px_batch* out, int32_t* d_out_seg, int64_t* d_ngroups,
                            void* d_ws, size_t ws_bytes, void* stream) {
    CallRange nvtx_range("px_join_probe_agg");
    set_error("");
    px_status s = check_batch(probe, "px_join_probe_agg probe");
    if (s != PX_OK) return s;
    if (!d_table || !aligned16(d_table)) return fail(PX_ERR_INVALID, "px_join_probe_agg: null or misaligned table");
    if (fk_col < 0 || fk_col >= probe->ncols || probe->cols[fk_col].type != PX_I64)
        return fail(PX_ERR_INVALID, "px_join_probe_agg: fk_col must name a PX_I64 probe column");
    if (!group || nbuild < 0) return fail(PX_ERR_INVALID, "px_join_probe_agg: group column");
    s = check_col(group, "px_join_probe_agg group", nbuild == 0);
    if (s != PX_OK) return s;
    if (group_hi < group_lo) return fail(PX_ERR_INVALID, "px_join_probe_agg: empty group range");
    px_key_range r = {};
    r.lo[0] = group_lo;
    r.hi[0] = group_hi;
    const int32_t key0 = 0;
    const ProbeSrc ps = {d_table, fk_col, group, nbuild};
    return groupby_impl(probe, &key0, 1, aggs, naggs, d_sel, d_nsel, d_seg, nsegs, &r, max_groups, out, d_out_seg,
                        d_ngroups, 0, d_ws, ws_bytes, stream, &ps);
}

}  // extern "C"

// Selection over materialised metrics in one launch (constraint filter + top-k / Pareto front of
// Sec. 3.2 / Sec. 4.1 on arrays written by guide_simulate).
//
// A selection keeps a handful of configs out of many, so what bounds it is a chain of latencies, not
// bandwidth: on a million configs the arrays are read in 3 us, and everything else is steps that wait
// for one another.  The steps are therefore parts of one cooperative kernel with grid barriers
// between them instead of five launches:
//
//   sample : rows of 64 consecutive configs, one out of every r at a hashed position (r = 1: all of
//            them), at most four per warp.  Their keys stay in registers.
//   bound  : top-k: the smallest pair of every group of warps goes to the workspace; after a barrier
//            every block works out for itself a pair that at least k of those are within (one
//            histogram of the encoded keys).  With r > 1 the sample pairs within it are gathered and
//            give, in the same way, a bound close to the sample's own k-th pair.  Pareto: the extreme
//            points of eight directions, over the lane, the warp, the block and, after a barrier, all
//            blocks ("killers"); over long ranges, after another one, a staircase of the sample's points.
//   filter : a config survives if it passes the constraints and its pair is within the bound, or no
//            killer strictly dominates it.  With r = 1 the values are still in registers, otherwise
//            one pass over the arrays.  Survivors go to a list in the workspace.
//   finish : the (few) survivors are ranked and the answer is written, by one block unless a front has
//            many of them.
//
// Bound and killers only exclude configs that cannot be part of the answer, whatever the sample
// looked like.  If the top-k list overflows, the k-th pair is closed in on by counting and the filter
// runs again.  A Pareto list of many goes through a staircase of its own points, as do the arrays again when
// it overflowed; only when it overflows a second time (fronts beyond the most a call reports, or thousands of equal
// points) the redo flag is raised and the accumulator kernel queued behind (select.cu) redoes the call.
//
// Ranges of up to 2048 configs are one block: its barriers are block barriers and nothing goes
// through the workspace.
//
// Blocks per SM: ranges whose rows all fit the warps' registers (1.2 M configs) take two, and their kernels have no
// pass over the arrays in them (WHOLE: half the code, 983,040 configs 25 -> 18 us top-k).  Longer
// ranges take one.  A cooperative launch starts only when all of its blocks have room, so with two per SM two
// selections on two streams run one after the other: 16.8 M configs, sweep and both selections, 334 us against 285
// with one, 2.2 M 124 against 100.  On one stream one block per SM costs nothing that a pass with more in flight does
// not give back (16.8 M: 64 + 79 us with two, 66 + 80 with one; 2.2 M: 33 + 39 and 33 + 34).
//
// Top-k + front on a B200 against chains of kernels (sample, refined bound, filter, rank, gated fallback): 983,040
// configs 18 + 25 us instead of 35 + 34; 30,720 configs 17 + 17 instead of 68 + 42; 16.8 M 66 + 80 instead of 65 + 83.
// Fronts of two continuous metrics (14.7 M): TTFT against cost per token 88 instead of 123, TTFT against throughput 92
// instead of 195; eight killers alone let more through than the list holds, and the call was done twice (588, 560).
#include <algorithm>
#include <atomic>
#include <cmath>

#include <cooperative_groups.h>

#include "select_src.cuh"

namespace guide {

static constexpr u32 CO_THREADS = 512, CO_WARPS = CO_THREADS / 32;
static constexpr u32 CO_BLOCKS_PER_SM = 2;      // 64 registers: 32 warps per SM, of one call or of two side by side
static constexpr u32 CO_ROWS = 4;               // sample rows a warp keeps in registers
static constexpr u32 CO_ONE_BLOCK_ROWS = 32;    // ranges up to this many rows are one block; its survivors stay in shared memory
static constexpr u32 CO_BOUND_LIST = 1024;      // most pairs a bound is worked out from: group minima, sample pairs within the coarse bound
static constexpr u32 CO_LIST = 2560;            // pairs the finishing block holds in shared memory (five per thread)
static constexpr u32 CO_BINS = 2 * CO_THREADS;  // bins of a histogram
static constexpr u32 CO_RANKED = 256;           // pairs the finishing block ranks by counting (at least two threads each)
static constexpr u32 CO_DIRS = 8;               // killers of a Pareto call
static constexpr u32 CO_P_DIRECT = 128;         // survivors one block compares all against all
static constexpr u32 CO_P_REFINE = 1024;        // more survivors than these are filtered once more
static constexpr u32 CO_STEPS = 2 * CO_THREADS; // steps of a staircase
static constexpr u32 CO_STAIR_RATIO = 12;       // the sample makes a staircase from one row of so many on (7 M configs): it costs
                                                // 3-6 us and saves the filter a second pass (14.7 M, TTFT against throughput: 89 us
                                                // with, 240 without; 4.2 M, latency against cost: 44 with, 39 without)
static constexpr u32 CO_P_CHUNK = 1024;         // survivors staged in shared memory at a time
static constexpr u32 CO_MAX_BLOCKS = 512;       // workspace for the blocks' killer candidates
static_assert(CO_ONE_BLOCK_ROWS * ROW <= CO_LIST && CO_LIST % CO_THREADS == 0, "one block's whole range fits its list");

template <int NA>
struct CoopSrc {
    Arr a[NA];        // entry 0 is the key (top-k) or x (Pareto), entry 1 is y (Pareto only)
    const uint8_t *status;
    int vec;          // every array is 16-byte aligned, status 4-byte (2: 16-byte too); 0: no wide loads
    // the bounds once more, as one comparison each: v, its sign flipped by flip, is at most bnd (unless free)
    double bnd[NA];
    u32 flip[NA], free[NA];
};

__device__ __forceinline__ double flipped(double v, u32 mask) { return __hiloint2double(__double2hiint(v) ^ (int)mask, __double2loint(v)); }
// the high half of metric_key, or, for a zero of the other sign, a little less
__device__ __forceinline__ u32 metric_key_high(const Arr &a, double v) {
    const u32 h = (u32)__double2hiint(v) ^ (a.neg ? 0x80000000u : 0u);
    return h ^ ((u32)((int)h >> 31) | 0x80000000u);
}

// The sample: groups of r consecutive rows, one row of each, at a hashed offset so that it does not
// lock onto a period of the config index.
struct Walk {
    u64 n_rows, n_slots;
    u32 r;
    __device__ __forceinline__ u64 row(u64 slot) const {
        if (r == 1) return slot;
        const u32 h = ((u32)slot * 2654435761u) >> 7;
        return slot * r + h % r;
    }
};

// status and values of this lane's two configs of a row; outside the range: status 0xFF.  LAST: not read again
// (marked for early eviction: with the lines kept, the sweep that overwrites the arrays next takes 8 of 68 us longer).
template <bool LAST, int NA>
__device__ __forceinline__ void load_row(const CoopSrc<NA> &s, u64 count, u64 row, bool live, u32 lane, u32 &st, double2 (&v)[NA]) {
    const u64 j = row * ROW + 2 * lane;
    if (live && s.vec && (row + 1) * ROW <= count) {
        const unsigned short *sp = reinterpret_cast<const unsigned short *>(s.status + j);
        st = LAST ? __ldcs(sp) : __ldcg(sp);
#pragma unroll
        for (int a = 0; a < NA; a++) {
            const double2 *vp = reinterpret_cast<const double2 *>(s.a[a].p + j);
            v[a] = LAST ? __ldcs(vp) : __ldcg(vp);
        }
    } else {
        const bool in0 = live && j < count, in1 = live && j + 1 < count;
        st = (in0 ? (u32)s.status[j] : 0xFFu) | ((in1 ? (u32)s.status[j + 1] : 0xFFu) << 8);
#pragma unroll
        for (int a = 0; a < NA; a++) {
            v[a].x = in0 ? s.a[a].p[j] : 0.0;
            v[a].y = in1 ? s.a[a].p[j + 1] : 0.0;
        }
    }
}

template <int NA>
__device__ __forceinline__ void row_ok(const CoopSrc<NA> &s, u32 st, const double2 (&v)[NA], bool &ok0, bool &ok1) {
    ok0 = (st & 0xFFu) == 0;
    ok1 = (st >> 8) == 0;
#pragma unroll
    for (int a = 0; a < NA; a++) {                     // a NaN fails an active bound
        ok0 &= s.free[a] || flipped(v[a].x, s.flip[a]) <= s.bnd[a];
        ok1 &= s.free[a] || flipped(v[a].y, s.flip[a]) <= s.bnd[a];
    }
}

// ---- a pass over everything ---------------------------------------------------------------------------
//
// Chunks of CO_CHUNK rows, from the end of the range backwards (when the metrics were written just before this call the
// end of the arrays is what the L2 still holds).  Every warp starts with three of its own; the others are taken
// through a counter in the workspace as warps get to them: rows that fit come in runs, and a chunk of live rows
// costs many times one without.
//
// A chunk's status bytes are one 16-byte load per lane, asked for two chunks ahead; values are loaded for rows with a
// config that passed its memory check only, which most rows of a large sweep have not, several such rows at a time,
// and looked at together.  That keeps enough in flight for one block of 16 warps per SM, so that two selections on
// two streams run side by side.
static constexpr u32 CO_CHUNK = 8;
template <int NA> __host__ __device__ constexpr int group_rows() { return NA <= 2 ? 4 : 2; }   // rows whose values are in flight at a time

struct ChunkWalk {
    u64 n_rows, chunk;                                 // chunk: number from the end, or past the last one
    // row u of the chunk; past the end of the walk: a huge number
    __device__ __forceinline__ u64 row(u32 u) const { return n_rows - 1 - (chunk * CO_CHUNK + u); }
    __device__ __forceinline__ bool more() const { return chunk * CO_CHUNK < n_rows; }
};

// status of 16 consecutive configs of a row (lane L: part L % 4 of row L / 4 of the chunk); outside the range: 0xFF
template <int NA>
__device__ __forceinline__ uint4 chunk_status(const CoopSrc<NA> &s, u64 count, const ChunkWalk &w, u32 lane) {
    uint4 st = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
    const u64 row = w.row(lane >> 2);
    if (row >= w.n_rows) return st;
    const u64 j = row * ROW + 16 * (lane & 3);
    if (s.vec && j + 16 <= count) {
        if (s.vec == 2) return __ldcs(reinterpret_cast<const uint4 *>(s.status + j));
        const u32 *q = reinterpret_cast<const u32 *>(s.status + j);
        return make_uint4(__ldcs(q), __ldcs(q + 1), __ldcs(q + 2), __ldcs(q + 3));
    }
    u32 wd[4];
#pragma unroll
    for (u32 i = 0; i < 4; i++) {
        wd[i] = 0;
#pragma unroll
        for (u32 k = 0; k < 4; k++) wd[i] |= (j + 4 * i + k < count ? (u32)s.status[j + 4 * i + k] : 0xFFu) << (8 * k);
    }
    return make_uint4(wd[0], wd[1], wd[2], wd[3]);
}
__device__ __forceinline__ bool has_zero_byte(u32 w) { return __vcmpeq4(w, 0u) != 0; }

// each(j, v, ok) for groups of rows that have a config to look at, by whole warps: the lane's two configs of row g are
// entries j[g] and j[g] + 1 of the arrays, v[g] their values; bits 2 g and 2 g + 1 of ok: they pass the constraints.
// counter: a word of the workspace, 0 on entry.
template <int NA, class Each>
__device__ __forceinline__ void for_live_rows(const CoopSrc<NA> &s, u64 count, u64 n_rows, u32 lane, u32 warp, u32 *counter, Each each) {
    constexpr int GROUP = group_rows<NA>();
    const u32 warps = gridDim.x * CO_WARPS;
    ChunkWalk w{n_rows, (u64)warp * gridDim.x + blockIdx.x}, w1{n_rows, w.chunk + warps}, w2{n_rows, w.chunk + 2 * (u64)warps};
    uint4 st = chunk_status(s, count, w, lane), st1 = chunk_status(s, count, w1, lane), st2 = chunk_status(s, count, w2, lane);
    while (w.more()) {
        u32 ticket = 0;
        if (lane == 0 && w2.more()) ticket = atomicAdd(counter, 1u);
        u32 live = __ballot_sync(0xFFFFFFFFu, has_zero_byte(st.x) | has_zero_byte(st.y) | has_zero_byte(st.z) | has_zero_byte(st.w));
        live |= live >> 1;
        live = (live | live >> 2) & 0x11111111u;       // bit 4 u: row u
        while (live) {
            double2 v[GROUP][NA];
            u64 j[GROUP];
            u32 st_v[GROUP], ok = 0;
#pragma unroll
            for (int g = 0; g < GROUP; g++) {
                const u64 row = w.row(((u32)__ffs(live) - 1) >> 2);
                j[g] = row * ROW + 2 * lane;
                load_row<true>(s, count, row, live != 0, lane, st_v[g], v[g]);
                live &= live - 1;
            }
#pragma unroll
            for (int g = 0; g < GROUP; g++) {
                bool ok0, ok1;
                row_ok(s, st_v[g], v[g], ok0, ok1);
                ok |= (ok0 ? 1u : 0u) << (2 * g) | (ok1 ? 1u : 0u) << (2 * g + 1);
            }
            each(j, v, ok);
        }
        w = w1; w1 = w2; st = st1; st1 = st2;
        w2.chunk = w1.more() ? 3 * (u64)warps + __shfl_sync(0xFFFFFFFFu, ticket, 0) : w1.chunk;     // past the end: stays there
        st2 = chunk_status(s, count, w2, lane);
    }
}

__device__ __forceinline__ void grid_barrier() {
    if (gridDim.x == 1) __syncthreads();
    else cooperative_groups::this_grid().sync();
}

// ---- block-wide counting --------------------------------------------------------------------------

struct CountScratch {
    u32 part[2][CO_WARPS];
    u64 lo[CO_WARPS], hi[CO_WARPS];
};

// Sum over the block.  Two buffers in turn: one barrier per call is enough.
__device__ __forceinline__ u32 block_sum(u32 v, u32 (*part)[CO_WARPS], u32 &phase) {
    const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = __reduce_add_sync(0xFFFFFFFFu, v);
    if (lane == 0) part[phase][warp] = v;
    __syncthreads();
    const u32 t = lane < CO_WARPS ? part[phase][lane] : 0u;
    phase ^= 1;
    return __reduce_add_sync(0xFFFFFFFFu, t);
}

__device__ __forceinline__ void block_min_max(u64 &lo, u64 &hi, u64 *slo, u64 *shi) {
    const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int d = 16; d > 0; d >>= 1) {
        const u64 ol = __shfl_xor_sync(0xFFFFFFFFu, lo, d), oh = __shfl_xor_sync(0xFFFFFFFFu, hi, d);
        lo = ol < lo ? ol : lo; hi = oh > hi ? oh : hi;
    }
    __syncthreads();                                   // earlier readers of the scratch are done
    if (lane == 0) { slo[warp] = lo; shi[warp] = hi; }
    __syncthreads();
    for (u32 w = 0; w < CO_WARPS; w++) { lo = slo[w] < lo ? slo[w] : lo; hi = shi[w] > hi ? shi[w] : hi; }
}

// A pair (bkey, bidx) that at least k and, ties or not, at most k + slack of the block's pairs are
// within (the total order is (key, index); indices are distinct).  A bisection on the encoded key,
// then, if one key is shared by too many, on the index; it stops as soon as the count is in the
// window.  Entries with an all-ones index are padding.  All-ones when there are fewer than k pairs.
// Collective; every thread gets the result.
template <u32 PER>
__device__ __noinline__ void kth_bound(const u64 (&key)[PER], const u64 (&idx)[PER], u32 k, u32 slack, CountScratch &sc, u64 &bkey,
                                       u64 &bidx) {
    u32 phase = 0;
    __syncthreads();                                   // the scratch is free
    u32 n = 0;
    u64 lo = KEY_MAX, hi = 0;
#pragma unroll
    for (u32 u = 0; u < PER; u++)
        if (idx[u] != KEY_MAX) { n++; lo = key[u] < lo ? key[u] : lo; hi = key[u] > hi ? key[u] : hi; }
    bkey = KEY_MAX; bidx = KEY_MAX;
    if (block_sum(n, sc.part, phase) < k) return;
    block_min_max(lo, hi, sc.lo, sc.hi);
    while (lo < hi) {
        const u64 mid = lo + ((hi - lo) >> 1);
        u32 c = 0;
#pragma unroll
        for (u32 u = 0; u < PER; u++) c += (idx[u] != KEY_MAX && key[u] <= mid) ? 1u : 0u;
        c = block_sum(c, sc.part, phase);
        if (c < k) { lo = mid + 1; continue; }
        hi = mid;
        if (c <= k + slack) { bkey = hi; return; }
    }
    bkey = hi;                                         // the k-th key itself; maybe many share it
    u32 c = 0;
    u64 ilo = KEY_MAX, ihi = 0;
#pragma unroll
    for (u32 u = 0; u < PER; u++) {
        if (idx[u] == KEY_MAX) continue;
        c += key[u] <= bkey ? 1u : 0u;
        if (key[u] == bkey) { ilo = idx[u] < ilo ? idx[u] : ilo; ihi = idx[u] > ihi ? idx[u] : ihi; }
    }
    if (block_sum(c, sc.part, phase) <= k + slack) return;
    block_min_max(ilo, ihi, sc.lo, sc.hi);
    while (ilo < ihi) {
        const u64 mid = ilo + ((ihi - ilo) >> 1);
        c = 0;
#pragma unroll
        for (u32 u = 0; u < PER; u++) c += (idx[u] != KEY_MAX && pair_le(key[u], idx[u], bkey, mid)) ? 1u : 0u;
        c = block_sum(c, sc.part, phase);
        if (c < k) { ilo = mid + 1; continue; }
        ihi = mid;
        if (c <= k + slack) break;
    }
    bidx = ihi;
}

// The same from one histogram of the keys' high halves, which as a rule decides: four barriers instead
// of one per round.  Where the bin of the k-th pair takes the count above k + slack (many keys
// share it) the bisection follows.  All-ones when there are fewer than k pairs.
template <u32 PER>
__device__ __forceinline__ void histogram_bound(const u64 (&key)[PER], const u64 (&idx)[PER], u32 k, u32 slack, u32 *bins, CountScratch &sc,
                                                u64 &bkey, u64 &bidx) {
    const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5, FULL = 0xFFFFFFFFu;
    __syncthreads();                                   // the scratch is free
    u32 lo = FULL, hi = 0;
#pragma unroll
    for (u32 u = 0; u < PER; u++)
        if (idx[u] != KEY_MAX) { const u32 h = (u32)(key[u] >> 32); lo = min(lo, h); hi = max(hi, h); }
    lo = __reduce_min_sync(FULL, lo); hi = __reduce_max_sync(FULL, hi);
    if (lane == 0) { sc.part[0][warp] = lo; sc.part[1][warp] = hi; }
    for (u32 i = threadIdx.x; i < CO_BINS; i += CO_THREADS) bins[i] = 0;
    if (threadIdx.x == 0) { sc.lo[0] = KEY_MAX; sc.hi[0] = 0; }
    __syncthreads();
    lo = __reduce_min_sync(FULL, sc.part[0][lane % CO_WARPS]); hi = __reduce_max_sync(FULL, sc.part[1][lane % CO_WARPS]);
    const u32 range = hi >= lo ? hi - lo : 0, width = 32 - __clz(range | 1u), shift = width > 10 ? width - 10 : 0;   // range >> shift < 1024
    static_assert(CO_BINS == 1024, "ten bits of the range");
#pragma unroll
    for (u32 u = 0; u < PER; u++)
        if (idx[u] != KEY_MAX) atomicAdd(&bins[((u32)(key[u] >> 32) - lo) >> shift], 1u);
    __syncthreads();
    const u32 b0 = bins[2 * threadIdx.x], b1 = bins[2 * threadIdx.x + 1];
    u32 incl = b0 + b1;
    for (u32 d = 1; d < 32; d <<= 1) {
        const u32 o = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) sc.part[0][warp] = incl;
    __syncthreads();
    u32 off = 0;
    for (u32 w = 0; w < warp; w++) off += sc.part[0][w];
    incl += off;
    const u32 before = incl - b0 - b1;
    if (before < k && incl >= k) {                     // one thread: the k-th pair is in one of its two bins
        const bool first = before + b0 >= k;
        const u64 end = (u64)lo + ((u64)(2 * threadIdx.x + (first ? 1 : 2)) << shift);
        sc.lo[0] = end > FULL ? KEY_MAX : (end << 32) - 1;
        sc.hi[0] = first ? before + b0 : incl;
    }
    __syncthreads();
    bkey = sc.lo[0]; bidx = KEY_MAX;
    const u32 c = (u32)sc.hi[0];
    if (c > k + slack) kth_bound<PER>(key, idx, k, slack, sc, bkey, bidx);
}

// ... of n pairs of a list in the workspace (of PER per thread spread over it, if it is longer)
template <u32 PER>
__device__ __forceinline__ void list_bound(const KI *list, u32 n, u32 k, u32 *bins, CountScratch &sc, u64 &bkey, u64 &bidx) {
    constexpr u32 MOST = PER * CO_THREADS;
    const u32 step = n > MOST ? n / MOST : 1;
    u64 key[PER], idx[PER];
#pragma unroll
    for (u32 u = 0; u < PER; u++) {
        const u32 i = threadIdx.x + u * CO_THREADS;
        ulonglong2 e; e.x = KEY_MAX; e.y = KEY_MAX;
        if (i < min(n, MOST)) e = __ldcg(reinterpret_cast<const ulonglong2 *>(list + (size_t)i * step));
        key[u] = e.x; idx[u] = e.y;
    }
    histogram_bound<PER>(key, idx, k, k + 8, bins, sc, bkey, bidx);
}

// the takers of a warp append to a list through one atomic; entries beyond cap are counted, not stored
template <class T>
__device__ __forceinline__ void warp_append(bool take, const T &e, u32 *counter, T *list, u32 cap) {
    const u32 ballot = __ballot_sync(0xFFFFFFFFu, take);
    if (!ballot) return;
    const u32 lane = threadIdx.x & 31;
    u32 base = 0;
    if (lane == 0) base = atomicAdd(counter, __popc(ballot));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    const u32 pos = base + __popc(ballot & ((1u << lane) - 1));
    if (take && pos < cap) list[pos] = e;
}

// ---- top-k -------------------------------------------------------------------------------------------

struct FinishScratch {
    KI sl[CO_LIST];
    u32 bins[CO_BINS];
    u32 n;
};

// One block: the k smallest of n pairs, in order; of the list in the workspace, or (cand null) already in f.sl.
__device__ __noinline__ void topk_finish(const KI *cand, u32 n, u32 k, FinishScratch &f, CountScratch &sc, int negate, u64 *idx_out,
                                         double *key_out, u32 *count_out) {
    constexpr u32 PER = CO_LIST / CO_THREADS;
    const u32 found = min(n, k);
    if (threadIdx.x == 0) *count_out = found;
    for (u32 i = found + threadIdx.x; i < k; i += CO_THREADS) {
        idx_out[i] = KEY_MAX;
        key_out[i] = __longlong_as_double(0x7FF0000000000000LL);
    }
    if (n == 0) return;
    u32 c = n;
    u64 bkey = KEY_MAX, bidx = KEY_MAX;
    if (cand && n <= CO_LIST) {
        for (u32 i = threadIdx.x; i < n; i += CO_THREADS) {
            const ulonglong2 w = __ldcg(reinterpret_cast<const ulonglong2 *>(cand + i));
            f.sl[i].key = w.x; f.sl[i].idx = w.y;
        }
        __syncthreads();
    }
    // down to CO_RANKED pairs, and once towards the k that are wanted (ranking 232 pairs takes 10 us, 70 take 3): those
    // within a bound of what shared memory holds.  A list that does not fit it is gone through again with that bound,
    // which leaves out most of what was looked at.
    for (bool cut = false; c > CO_RANKED || (!cut && c > found + CO_RANKED / 4); cut = true) {
        if (c > CO_LIST) {
            __syncthreads();
            if (threadIdx.x == 0) f.n = 0;
            __syncthreads();
            for (u32 i0 = 0; i0 < n; i0 += CO_THREADS) {
                const u32 i = i0 + threadIdx.x;
                KI e; e.key = KEY_MAX; e.idx = KEY_MAX;
                if (i < n) {
                    const ulonglong2 w = __ldcg(reinterpret_cast<const ulonglong2 *>(cand + i));
                    e.key = w.x; e.idx = w.y;
                }
                warp_append(i < n && pair_le(e.key, e.idx, bkey, bidx), e, &f.n, f.sl, CO_LIST);
            }
            __syncthreads();
            c = f.n;
            if (c <= CO_RANKED) break;
        }
        u64 key[PER], idx[PER];
#pragma unroll
        for (u32 u = 0; u < PER; u++) {
            const u32 i = threadIdx.x + u * CO_THREADS;
            key[u] = KEY_MAX; idx[u] = KEY_MAX;
            if (i < min(c, CO_LIST)) { key[u] = f.sl[i].key; idx[u] = f.sl[i].idx; }
        }
        histogram_bound<PER>(key, idx, found, CO_RANKED - found, f.bins, sc, bkey, bidx);
        if (c > CO_LIST) continue;
        __syncthreads();
        if (threadIdx.x == 0) f.n = 0;
        __syncthreads();
#pragma unroll
        for (u32 u = 0; u < PER; u++) {
            KI e; e.key = key[u]; e.idx = idx[u];
            warp_append(idx[u] != KEY_MAX && pair_le(key[u], idx[u], bkey, bidx), e, &f.n, f.sl, CO_LIST);
        }
        __syncthreads();
        c = f.n;
    }
    // rank by counting: a power of two of threads per pair shares out the comparisons
    u32 tpe = 32;
    while (tpe * c > CO_THREADS) tpe >>= 1;            // c <= CO_RANKED: at least two
    const u32 me_i = threadIdx.x / tpe, part = threadIdx.x % tpe;
    const KI me = f.sl[min(me_i, c - 1)];
    u32 ahead = 0;
    for (u32 q = part; q < c; q += tpe) ahead += ki_less(f.sl[q], me) ? 1u : 0u;
    for (u32 d = tpe >> 1; d > 0; d >>= 1) ahead += __shfl_xor_sync(0xFFFFFFFFu, ahead, d);
    if (part == 0 && me_i < c && ahead < k) {
        const double v = dec(me.key);
        idx_out[ahead] = me.idx;
        key_out[ahead] = negate ? 0.0 - v : v;
    }
}

// the passing pairs within a bound, appended to a list
template <int NA>
__device__ __forceinline__ void topk_filter(const CoopSrc<NA> &s, const Range &r, u64 n_rows, u32 *ticket, u64 bkey, u64 bidx, u32 *count, KI *cand) {
    // first by the bound's value: what compares greater has a greater key (a NaN does not compare)
    const double bval = dec(bkey);
    const u32 neg = s.a[0].neg ? 0x80000000u : 0u;
    for_live_rows<NA>(s, r.count, n_rows, threadIdx.x & 31, threadIdx.x >> 5, ticket, [&](const u64 *j, const double2 (*v)[NA], u32 pass) {
#pragma unroll
        for (int g = 0; g < group_rows<NA>(); g++) {
            if (flipped(v[g][0].x, neg) > bval) pass &= ~(1u << (2 * g));
            if (flipped(v[g][0].y, neg) > bval) pass &= ~(2u << (2 * g));
        }
        if (!__any_sync(0xFFFFFFFFu, pass)) return;                    // the usual case
#pragma unroll
        for (int i = 0; i < 2 * group_rows<NA>(); i++) {
            KI e;
            e.key = metric_key(s.a[0], (i & 1) ? v[i >> 1][0].y : v[i >> 1][0].x); e.idx = r.first + j[i >> 1] + (i & 1);
            warp_append(((pass >> i) & 1u) && pair_le(e.key, e.idx, bkey, bidx), e, count, cand, TK_CAND_CAP);
        }
    });
}

// The survivors did not fit their list (the sample had too few passing configs, or none of the better ones).  The k-th
// pair is then closed in on by counting: every pass makes a histogram of the passing keys in [lo, hi] over the
// whole grid, and [lo, hi] becomes the bin the k-th of them is in: ten bits a pass, seven passes at most, and four or five
// on the index where one key alone is too many.  It ends as soon as the pairs up to that bin's end fit the
// list; one more pass collects them.  (Tightening the bound by what the list holds takes as many passes as the
// list goes into the passing configs when those are met worst first.)
// Collective over the grid; khi: the bound's key.  gbins: two histograms in the workspace.  Returns the new count.
template <int NA>
__device__ __noinline__ u32 topk_overflow(const CoopSrc<NA> s, const Range r, u64 n_rows, u32 k, u32 *header, unsigned long long *gbins,
                                          KI *cand, u32 *bins, CountScratch &sc, u64 khi) {
    static_assert(CO_BINS == 1024 && 2 * CO_BINS * sizeof(u64) <= CO_BOUND_LIST * sizeof(KI), "ten bits; two histograms in the minima's place");
    const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5, FULL = 0xFFFFFFFFu;
    u64 lo = 0, hi = khi, kkey = 0, before = 0;        // before: passing pairs below lo
    bool by_idx = false;                               // [lo, hi] are indices of configs with key kkey
    u32 *ticket;
    for (u32 pass = 0;; pass++) {
        unsigned long long *g = gbins + (pass & 1) * CO_BINS;           // last read two passes ago, as the ticket
        ticket = header + ((pass & 1) ? TK_TICKET : TK_TICKET2);
        for (u32 i = blockIdx.x * CO_THREADS + threadIdx.x; i < CO_BINS; i += gridDim.x * CO_THREADS) g[i] = 0;
        if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0;
        for (u32 i = threadIdx.x; i < CO_BINS; i += CO_THREADS) bins[i] = 0;
        grid_barrier();
        const u32 width = 64 - __clzll((long long)((hi - lo) | 1ull)), shift = width > 10 ? width - 10 : 0;
        for_live_rows<NA>(s, r.count, n_rows, lane, warp, ticket, [&](const u64 *j, const double2 (*v)[NA], u32 ok) {
#pragma unroll
            for (int i = 0; i < 2 * group_rows<NA>(); i++) {
                const u64 key = metric_key(s.a[0], (i & 1) ? v[i >> 1][0].y : v[i >> 1][0].x), idx = r.first + j[i >> 1] + (i & 1);
                const u64 at = by_idx ? idx : key;
                if (((ok >> i) & 1u) && at >= lo && at <= hi && (!by_idx || key == kkey)) atomicAdd(&bins[(at - lo) >> shift], 1u);
            }
        });
        __syncthreads();
        for (u32 i = threadIdx.x; i < CO_BINS; i += CO_THREADS)
            if (bins[i]) atomicAdd(g + i, (unsigned long long)bins[i]);
        grid_barrier();
        // the bin of the k-th pair: two bins per thread
        const u64 b0 = __ldcg(g + 2 * threadIdx.x), b1 = __ldcg(g + 2 * threadIdx.x + 1);
        u64 incl = b0 + b1;
        for (u32 d = 1; d < 32; d <<= 1) {
            const u64 o = __shfl_up_sync(FULL, incl, d);
            if (lane >= d) incl += o;
        }
        if (lane == 31) sc.lo[warp] = incl;
        __syncthreads();
        u64 off = before;
        for (u32 q = 0; q < warp; q++) off += sc.lo[q];
        incl += off;
        const u64 prev = incl - b0 - b1;
        __syncthreads();
        if (prev < k && incl >= k) {                   // one thread
            const bool first = prev + b0 >= k;
            sc.hi[0] = 2 * threadIdx.x + (first ? 0 : 1);              // the bin
            sc.hi[1] = first ? prev : prev + b0;                       // pairs below it
            sc.hi[2] = first ? prev + b0 : incl;                       // ... and up to its end
        }
        __syncthreads();
        const u64 upto = sc.hi[2], span = (1ull << shift) - 1;
        before = sc.hi[1];
        lo += sc.hi[0] << shift;
        hi = hi - lo <= span ? hi : lo + span;
        __syncthreads();
        if (upto <= TK_CAND_CAP) break;
        if (!by_idx && lo == hi) { by_idx = true; kkey = lo; lo = r.first; hi = r.first + r.count - 1; }
    }
    u32 *count = header + TK_COUNT2;                   // untouched so far
    ticket = ticket == header + TK_TICKET ? header + TK_TICKET2 : header + TK_TICKET;
    if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0;
    grid_barrier();
    topk_filter(s, r, n_rows, ticket, by_idx ? kkey : hi, by_idx ? hi : KEY_MAX, count, cand);
    grid_barrier();
    return __ldcg(count);
}

// WHOLE: the sample is everything (w.r == 1), and the one pass over the arrays is the sample's.
template <int NA, bool WHOLE>
__global__ void __launch_bounds__(CO_THREADS, CO_BLOCKS_PER_SM)
k_topk_coop(CoopSrc<NA> s, Range r, Walk w, u32 k, u32 group_log2, u32 *header, KI *minima, KI *spairs, KI *cand, int negate,
            u64 *idx_out, double *key_out, u32 *count_out) {
    __shared__ FinishScratch fin;
    __shared__ CountScratch sc;
    KI *sl = fin.sl;
    grid_dep_wait();
    const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // nothing reads the header before the first barrier
    if (blockIdx.x == 0 && threadIdx.x < 64) header[threadIdx.x] = 0;
    // ---- sample: this warp's rows; the groups of 2^group_log2 warps take rows far apart ----
    const u32 n_groups = (gridDim.x * CO_WARPS) >> group_log2;
    const u32 group = (blockIdx.x * CO_WARPS + warp) >> group_log2, member = warp & ((1u << group_log2) - 1);
    u64 key[2 * CO_ROWS];
    u32 ok = 0;
    {
        u32 st[CO_ROWS];
        double2 v[CO_ROWS][NA];
#pragma unroll
        for (u32 u = 0; u < CO_ROWS; u++) {
            const u64 slot = (u64)((u << group_log2) + member) * n_groups + group;
            load_row<false>(s, r.count, w.row(slot), slot < w.n_slots, lane, st[u], v[u]);
        }
#pragma unroll
        for (u32 u = 0; u < CO_ROWS; u++) {
            bool ok0, ok1;
            row_ok(s, st[u], v[u], ok0, ok1);
            key[2 * u] = metric_key(s.a[0], v[u][0].x);
            key[2 * u + 1] = metric_key(s.a[0], v[u][0].y);
            ok |= (ok0 ? 1u : 0u) << (2 * u) | (ok1 ? 1u : 0u) << (2 * u + 1);
        }
    }
    auto index_of = [&](u32 i) {                       // config index of sample value i of this lane
        const u64 slot = (u64)(((i >> 1) << group_log2) + member) * n_groups + group;
        return r.first + w.row(slot) * ROW + 2 * lane + (i & 1);
    };
    // ---- one block: what passes is ranked where it is ----
    if (WHOLE && gridDim.x == 1) {
        if (threadIdx.x == 0) fin.n = 0;
        __syncthreads();
#pragma unroll
        for (u32 i = 0; i < 2 * CO_ROWS; i++) {
            KI e; e.key = key[i]; e.idx = index_of(i);
            warp_append(((ok >> i) & 1u) != 0, e, &fin.n, sl, CO_LIST);
        }
        __syncthreads();
        const u32 n = fin.n;
        __syncthreads();
        topk_finish(nullptr, n, k, fin, sc, negate, idx_out, key_out, count_out);
        return;
    }
    // ---- coarse bound: the smallest pair of every group, then a pair k of them are within ----
    {
        u64 bk = KEY_MAX, bi = KEY_MAX;
#pragma unroll
        for (u32 i = 0; i < 2 * CO_ROWS; i++)
            if ((ok >> i) & 1u) pair_min(bk, bi, key[i], index_of(i));
        for (int d = 16; d > 0; d >>= 1)
            pair_min(bk, bi, __shfl_xor_sync(0xFFFFFFFFu, bk, d), __shfl_xor_sync(0xFFFFFFFFu, bi, d));
        if (lane == 0) { sl[warp].key = bk; sl[warp].idx = bi; }
        __syncthreads();
        if (threadIdx.x < (CO_WARPS >> group_log2)) {
            const KI *mine = sl + (threadIdx.x << group_log2);
            bk = mine[0].key; bi = mine[0].idx;
            for (u32 q = 1; q < (1u << group_log2); q++) pair_min(bk, bi, mine[q].key, mine[q].idx);
            ulonglong2 m; m.x = bk; m.y = bi;
            *reinterpret_cast<ulonglong2 *>(minima + ((blockIdx.x * CO_WARPS) >> group_log2) + threadIdx.x) = m;
        }
    }
    grid_barrier();
    u64 bkey, bidx;
    list_bound<CO_BOUND_LIST / CO_THREADS>(minima, n_groups, k, fin.bins, sc, bkey, bidx);
    // ---- the sample values within it: the survivors themselves, or (r > 1) the pairs of a closer bound ----
#pragma unroll
    for (u32 i = 0; i < 2 * CO_ROWS; i++) {
        KI e; e.key = key[i]; e.idx = index_of(i);
        const bool take = ((ok >> i) & 1u) && pair_le(e.key, e.idx, bkey, bidx);
        if (WHOLE) warp_append(take, e, header + TK_COUNT, cand, TK_CAND_CAP);
        else warp_append(take, e, header + TK_SAMPLED, spairs, CO_BOUND_LIST);
    }
    grid_barrier();
    if (!WHOLE) {
        // of more pairs than the list holds the stored ones still give a valid bound; fewer than k only
        // when the coarse bound is all-ones, which then stays
        const u32 ns = min(__ldcg(header + TK_SAMPLED), CO_BOUND_LIST);
        if (ns >= k) list_bound<CO_BOUND_LIST / CO_THREADS>(spairs, ns, k, fin.bins, sc, bkey, bidx);
    }
    // ---- filter: the sample's own survivors when it was everything, else one pass over the arrays ----
    if (!WHOLE) {
        topk_filter(s, r, w.n_rows, header + TK_TICKET, bkey, bidx, header + TK_COUNT, cand);
        grid_barrier();
    }
    u32 n = __ldcg(header + TK_COUNT);
    if (n > TK_CAND_CAP)
        n = topk_overflow(s, r, w.n_rows, k, header, reinterpret_cast<unsigned long long *>(minima), cand, fin.bins, sc, bkey);
    if (blockIdx.x == 0) topk_finish(cand, n, k, fin, sc, negate, idx_out, key_out, count_out);
}

// ---- Pareto ------------------------------------------------------------------------------------------

// The killers are the extreme points of a few directions: of the points seen, the one that minimises a
// weighted sum of the two encoded metrics (their high halves: about the logarithms).  Every one is a
// real point, so whatever it strictly dominates is out.  No direction is an axis: the other metric
// decides between points that share the best value of one, as they do where it has few values.
__device__ __forceinline__ u32 direction_weight(u32 d) { return d == 0 ? 31u : d == CO_DIRS - 1 ? 1u : 30u - 4u * d; }
static_assert(CO_DIRS == 8, "weights 31, 26, 22, 18, 14, 10, 6, 1 of 32");
// a missing point (all-ones twice) has the largest score there is
__device__ __forceinline__ u32 direction_score(u64 x, u64 y, u32 w) { return (u32)(x >> 37) * w + (u32)(y >> 37) * (32u - w); }

// is this the lane with the smallest score of the warp?
__device__ __forceinline__ bool warp_best(u32 score) {
    const u32 s = __reduce_min_sync(0xFFFFFFFFu, score);
    return (threadIdx.x & 31) == (u32)__ffs(__ballot_sync(0xFFFFFFFFu, score == s)) - 1;
}

struct Killers8 {
    const P2 *k;
    const uint2 *hi;                                   // their high halves, which decide nearly always
    // of n points, those whose high halves no killer's rule out (all bits of alive: the ones to ask about)
    template <int N>
    __device__ __forceinline__ u32 left(const u32 (&X)[N], const u32 (&Y)[N], u32 alive) const {
#pragma unroll
        for (u32 q = 0; q < CO_DIRS; q++) {
            const uint2 h = hi[q];
#pragma unroll
            for (int i = 0; i < N; i++)
                if (h.x < X[i] && h.y < Y[i]) alive &= ~(1u << i);
        }
        return alive;
    }
    // the same of one point
    __device__ __forceinline__ bool kills_high(u64 x, u64 y) const {
        const u32 X = (u32)(x >> 32), Y = (u32)(y >> 32);
        bool dead = false;
#pragma unroll
        for (u32 q = 0; q < CO_DIRS; q++) { const uint2 h = hi[q]; dead |= h.x < X && h.y < Y; }
        return dead;
    }
    // strictly dominated by one of them?
    __device__ __forceinline__ bool kills(u64 x, u64 y) const {
        bool dead = false;
#pragma unroll 1
        for (u32 q = 0; q < CO_DIRS; q++) dead |= dominates(k[q].x, k[q].y, x, y);
        return dead;
    }
};

// One block: the front of n points, by all-against-all comparison shared out over the threads, in
// ascending x (the x of a front are distinct).  flags: n bytes.
__device__ __noinline__ void pareto_small(const P3 *sv, u32 n, unsigned char *flags, u32 lim, u64 *idx_out, u32 *count_out) {
    u32 tpe = 32;
    while (tpe > 1 && tpe * n > CO_THREADS) tpe >>= 1;
    const u32 part = threadIdx.x % tpe, per_round = CO_THREADS / tpe;
    for (u32 g0 = 0; g0 < n; g0 += per_round) {
        const u32 g = g0 + threadIdx.x / tpe;
        const P3 me = sv[min(g, n - 1)];
        u32 out = 0;
        for (u32 q = part; q < n; q += tpe) {
            const P3 o = sv[q];
            out |= dominates(o.x, o.y, me.x, me.y) || (o.x == me.x && o.y == me.y && o.idx < me.idx) ? 1u : 0u;
        }
        for (u32 d = tpe >> 1; d > 0; d >>= 1) out |= __shfl_xor_sync(0xFFFFFFFFu, out, d);
        if (part == 0 && g < n) flags[g] = out ? 0 : 1;
    }
    __syncthreads();
    for (u32 g = threadIdx.x; g < n; g += CO_THREADS) {
        if (!flags[g]) continue;
        u32 ahead = 0;
        for (u32 q = 0; q < n; q++) ahead += flags[q] && sv[q].x < sv[g].x ? 1u : 0u;
        if (ahead < lim) idx_out[ahead] = sv[g].idx;
    }
    u32 total = 0;
    for (u32 g0 = 0; g0 < n; g0 += CO_THREADS) total += __syncthreads_count(g0 + threadIdx.x < n && flags[g0 + threadIdx.x]);
    if (threadIdx.x == 0) *count_out = total > GUIDE_PARETO_MAX ? 0xFFFFFFFFu : total;
}

// Eight points guard the hull of a front only: of two continuous metrics thousands of points behind its concave stretches
// survive them (TTFT against cost per token on 14.7 M configs 21,557, for a front of 42).  Behind them stands a
// staircase: the range of x between the killers in equal parts of the encoded metric (what is left and right of it
// apart), and on every step the smallest y of the points seen there.  A point with a y no smaller than one on a lower step
// is out: that one is real, and its x is smaller.
struct Staircase {
    u64 xlo, xhi;
    u32 shift;
    const u64 *low;                                    // shared: per step, the smallest y of all lower ones; null: no staircase
    __device__ __forceinline__ explicit Staircase(const Killers8 &K) : low(nullptr) {
        xlo = KEY_MAX; xhi = 0;
        for (u32 q = 0; q < CO_DIRS; q++) {
            const P2 p = K.k[q];
            if (p.x == KEY_MAX && p.y == KEY_MAX) continue;
            xlo = p.x < xlo ? p.x : xlo; xhi = p.x > xhi ? p.x : xhi;
        }
        if (xlo > xhi) { xlo = 0; xhi = KEY_MAX; }     // no killer: the sample had no passing config
        const u32 width = 64 - __clzll((long long)((xhi - xlo) | 1ull));
        shift = width > 10 ? width - 10 : 0;
    }
    __device__ __forceinline__ u32 step(u64 x) const {
        if (x <= xlo) return 0;
        if (x >= xhi) return CO_STEPS - 1;
        return 1 + ((u32)((x - xlo - 1) >> shift) * (CO_STEPS - 2) >> 10);
    }
    __device__ __forceinline__ void put(unsigned long long *g, u64 x, u64 y) const { atomicMin(g + step(x), y); }
    // after a barrier: g's minima into shared memory, each step with those of all lower ones
    __device__ __forceinline__ void read(const unsigned long long *g, u64 *steps, u64 *part) {
        static_assert(CO_STEPS == 2 * CO_THREADS, "two steps per thread");
        const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5, FULL = 0xFFFFFFFFu;
        const u64 e0 = __ldcg(g + 2 * threadIdx.x), e1 = __ldcg(g + 2 * threadIdx.x + 1);
        u64 incl = e0 < e1 ? e0 : e1;
        for (u32 d = 1; d < 32; d <<= 1) {
            const u64 o = __shfl_up_sync(FULL, incl, d);
            if (lane >= d && o < incl) incl = o;
        }
        if (lane == 31) part[warp] = incl;
        u64 below = __shfl_up_sync(FULL, incl, 1);
        if (lane == 0) below = KEY_MAX;
        __syncthreads();
        for (u32 q = 0; q < warp; q++) below = part[q] < below ? part[q] : below;
        steps[2 * threadIdx.x] = below;
        steps[2 * threadIdx.x + 1] = e0 < below ? e0 : below;
        __syncthreads();
        low = steps;
    }
    __device__ __forceinline__ bool behind(u64 x, u64 y) const {
        if (!low) return false;
        const u64 l = low[step(x)];
        return l <= y && l != KEY_MAX;
    }
};

// the passing points that no killer dominates and that are not behind the staircase, appended to a list
template <int NA>
__device__ __forceinline__ void pareto_filter(const CoopSrc<NA> &s, const Range &r, u64 n_rows, u32 *ticket, const Killers8 &K, const Staircase &S,
                                              u32 *count, P3 *surv) {
    for_live_rows<NA>(s, r.count, n_rows, threadIdx.x & 31, threadIdx.x >> 5, ticket, [&](const u64 *j, const double2 (*v)[NA], u32 pass) {
        constexpr int N = 2 * group_rows<NA>();
        u32 X[N], Y[N];
#pragma unroll
        for (int i = 0; i < N; i++) {
            const double2 *q = v[i >> 1];
            X[i] = metric_key_high(s.a[0], (i & 1) ? q[0].y : q[0].x);
            Y[i] = metric_key_high(s.a[1], (i & 1) ? q[1].y : q[1].x);
        }
        pass = K.left(X, Y, pass);
        if (!__any_sync(0xFFFFFFFFu, pass)) return;
#pragma unroll
        for (int i = 0; i < N; i++) {
            if (!__any_sync(0xFFFFFFFFu, (pass >> i) & 1u)) continue;
            const double2 *q = v[i >> 1];
            P3 e;
            e.x = metric_key(s.a[0], (i & 1) ? q[0].y : q[0].x); e.y = metric_key(s.a[1], (i & 1) ? q[1].y : q[1].x);
            e.idx = r.first + j[i >> 1] + (i & 1);
            warp_append(((pass >> i) & 1u) && !S.behind(e.x, e.y) && !K.kills(e.x, e.y), e, count, surv, PA_SURV_CAP);
        }
    });
}

// Still many survivors: they go into the staircase themselves, and it filters their list, or, when that overflowed, the
// arrays again (the stored part of the list still is made of real points).  Collective over the grid; steps and part: shared.
// Returns the new count.
template <int NA, bool WHOLE>
__device__ __noinline__ u32 pareto_refine(const CoopSrc<NA> s, const Range r, u64 n_rows, u32 n, u32 *header, const Killers8 K,
                                          unsigned long long *gsteps, const P3 *surv, P3 *kept, u64 *steps, u64 *part) {
    const u32 threads = gridDim.x * CO_THREADS, m = min(n, PA_SURV_CAP);
    const u64 *words = reinterpret_cast<const u64 *>(surv);
    Staircase S(K);
    if (WHOLE) {                                       // made here: few ranges this short need it
        if (blockIdx.x == 0) gsteps[threadIdx.x] = gsteps[threadIdx.x + CO_THREADS] = KEY_MAX;
        grid_barrier();
    }
    for (u32 i = blockIdx.x * CO_THREADS + threadIdx.x; i < m; i += threads)
        S.put(gsteps, __ldcg(words + 3 * (size_t)i), __ldcg(words + 3 * (size_t)i + 1));
    grid_barrier();
    S.read(gsteps, steps, part);
    if (n <= PA_SURV_CAP) {
        for (u32 i0 = blockIdx.x * CO_THREADS; i0 < m; i0 += threads) {
            const u32 i = i0 + threadIdx.x;
            P3 e; e.x = e.y = e.idx = 0;
            if (i < m) { e.x = __ldcg(words + 3 * (size_t)i); e.y = __ldcg(words + 3 * (size_t)i + 1); e.idx = __ldcg(words + 3 * (size_t)i + 2); }
            warp_append(i < m && !S.behind(e.x, e.y), e, header + PH_COUNT2, kept, PA_SURV_CAP);
        }
    } else {
        pareto_filter(s, r, n_rows, header + PH_TICKET2, K, S, header + PH_COUNT2, kept);
    }
    grid_barrier();
    return __ldcg(header + PH_COUNT2);
}

template <int NA, bool WHOLE>
__global__ void __launch_bounds__(CO_THREADS, CO_BLOCKS_PER_SM)
k_pareto_coop(CoopSrc<NA> s, Range r, Walk w, u32 *header, P2 *local, P3 *surv, P3 *kept, unsigned long long *gsteps, KI *front_list, u64 *idx_out,
              u32 out_cap, u32 *count_out) {
    __shared__ P3 sv[CO_P_CHUNK];
    __shared__ unsigned char flags[CO_P_CHUNK];
    __shared__ P2 best[CO_DIRS][CO_WARPS];
    __shared__ P2 ks[CO_DIRS];
    __shared__ uint2 kh[CO_DIRS];
    __shared__ u64 part[CO_WARPS];
    static_assert(sizeof(sv) >= CO_STEPS * sizeof(u64), "the steps' place until the finish");
    u64 *const steps = reinterpret_cast<u64 *>(sv);
    __shared__ u32 s_n;
    grid_dep_wait();
    const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // nothing reads these before the first barrier
    if (blockIdx.x == 0 && threadIdx.x < 64) header[threadIdx.x] = 0;
    if (!WHOLE && blockIdx.x == gridDim.x - 1) gsteps[threadIdx.x] = gsteps[threadIdx.x + CO_THREADS] = KEY_MAX;
    if (threadIdx.x == 0) s_n = 0;
    // ---- sample ----
    const u32 total_warps = gridDim.x * CO_WARPS, gwarp = blockIdx.x * CO_WARPS + warp;
    constexpr u32 N_PTS = 2 * CO_ROWS;
    u64 px[N_PTS], py[N_PTS];
    {
        u32 st[CO_ROWS];
        double2 v[CO_ROWS][NA];
#pragma unroll
        for (u32 u = 0; u < CO_ROWS; u++) {
            const u64 slot = (u64)u * total_warps + gwarp;
            load_row<false>(s, r.count, w.row(slot), slot < w.n_slots, lane, st[u], v[u]);
        }
#pragma unroll
        for (u32 u = 0; u < CO_ROWS; u++) {
            bool ok0, ok1;
            row_ok(s, st[u], v[u], ok0, ok1);
            px[2 * u] = py[2 * u] = px[2 * u + 1] = py[2 * u + 1] = KEY_MAX;       // "no point"
            if (ok0) { px[2 * u] = metric_key(s.a[0], v[u][0].x); py[2 * u] = metric_key(s.a[1], v[u][1].x); }
            if (ok1) { px[2 * u + 1] = metric_key(s.a[0], v[u][0].y); py[2 * u + 1] = metric_key(s.a[1], v[u][1].y); }
        }
    }
    // ---- killers: per direction the best point of the lane, the warp, the block, all blocks ----
#pragma unroll 2
    for (u32 d = 0; d < CO_DIRS; d++) {
        const u32 wd = direction_weight(d);
        u32 bs = 0xFFFFFFFFu;
        u64 bx = KEY_MAX, by = KEY_MAX;
#pragma unroll
        for (u32 i = 0; i < N_PTS; i++) {
            const u32 sc = direction_score(px[i], py[i], wd);
            if (sc < bs) { bs = sc; bx = px[i]; by = py[i]; }
        }
        if (warp_best(bs)) { best[d][warp].x = bx; best[d][warp].y = by; }
    }
    __syncthreads();
    if (warp < CO_DIRS) {
        P2 p; p.x = KEY_MAX; p.y = KEY_MAX;
        if (lane < CO_WARPS) p = best[warp][lane];
        if (warp_best(direction_score(p.x, p.y, direction_weight(warp)))) {
            if (WHOLE && gridDim.x == 1) {
                ks[warp] = p;
                kh[warp] = make_uint2((u32)(p.x >> 32), (u32)(p.y >> 32));
            } else {
                ulonglong2 e; e.x = p.x; e.y = p.y;
                *reinterpret_cast<ulonglong2 *>(local + (size_t)warp * CO_MAX_BLOCKS + blockIdx.x) = e;
            }
        }
    }
    if (!WHOLE || gridDim.x > 1) {
        static_assert(CO_WARPS == 2 * CO_DIRS, "two warps per direction");
        constexpr u32 PER = CO_MAX_BLOCKS / 64;
        grid_barrier();
        const u32 d = warp >> 1, wd = direction_weight(d);
        ulonglong2 e[PER];
#pragma unroll
        for (u32 u = 0; u < PER; u++) {
            const u32 b = (warp & 1) * 32 + lane + 64 * u;
            e[u].x = KEY_MAX; e[u].y = KEY_MAX;
            if (b < gridDim.x) e[u] = __ldcg(reinterpret_cast<const ulonglong2 *>(local + (size_t)d * CO_MAX_BLOCKS + b));
        }
        u32 bs = 0xFFFFFFFFu;
        u64 bx = KEY_MAX, by = KEY_MAX;
#pragma unroll
        for (u32 u = 0; u < PER; u++) {
            const u32 sc = direction_score(e[u].x, e[u].y, wd);
            if (sc < bs) { bs = sc; bx = e[u].x; by = e[u].y; }
        }
        if (warp_best(bs)) { best[d][warp & 1].x = bx; best[d][warp & 1].y = by; }
        __syncthreads();
        if (threadIdx.x < CO_DIRS) {
            const P2 a = best[threadIdx.x][0], b = best[threadIdx.x][1];
            const u32 wt = direction_weight(threadIdx.x);
            const P2 p = direction_score(b.x, b.y, wt) < direction_score(a.x, a.y, wt) ? b : a;
            ks[threadIdx.x] = p;
            kh[threadIdx.x] = make_uint2((u32)(p.x >> 32), (u32)(p.y >> 32));
        }
    }
    __syncthreads();
    const Killers8 K = {ks, kh};
    const u32 lim = min(out_cap, GUIDE_PARETO_MAX);
    // ---- filter: the sample itself when it was everything; else it makes the staircase, and one pass over the arrays ----
    if (WHOLE) {
#pragma unroll
        for (u32 i = 0; i < N_PTS; i++) {
            const bool real = !(px[i] == KEY_MAX && py[i] == KEY_MAX);
            if (!__any_sync(0xFFFFFFFFu, real)) continue;
            P3 e; e.x = px[i]; e.y = py[i];
            e.idx = r.first + ((u64)(i >> 1) * total_warps + gwarp) * ROW + 2 * lane + (i & 1);
            const bool take = real && !K.kills_high(px[i], py[i]) && !K.kills(px[i], py[i]);
            if (gridDim.x == 1) warp_append(take, e, &s_n, sv, CO_P_CHUNK);
            else warp_append(take, e, header + PH_COUNT, surv, PA_SURV_CAP);
        }
    } else {
        Staircase S(K);
        if (w.r >= CO_STAIR_RATIO) {
#pragma unroll
            for (u32 i = 0; i < N_PTS; i++)
                if (!(px[i] == KEY_MAX && py[i] == KEY_MAX) && !K.kills_high(px[i], py[i])) S.put(gsteps, px[i], py[i]);
            grid_barrier();
            S.read(gsteps, steps, part);
        }
        pareto_filter(s, r, w.n_rows, header + PH_TICKET, K, S, header + PH_COUNT, surv);
    }
    // ---- finish ----
    if (WHOLE && gridDim.x == 1) {
        __syncthreads();
        if (s_n > CO_P_CHUNK) { if (threadIdx.x == 0) header[1] = 1; }      // the general kernel redoes the call
        else pareto_small(sv, s_n, flags, lim, idx_out, count_out);
        return;
    }
    grid_barrier();
    u32 n = __ldcg(header + PH_COUNT);
    if (n > CO_P_REFINE) {
        n = pareto_refine<NA, WHOLE>(s, r, w.n_rows, n, header, K, gsteps, surv, kept, steps, part);
        surv = kept;
    }
    if (n > PA_SURV_CAP) {
        if (blockIdx.x == 0 && threadIdx.x == 0) header[1] = 1;
        return;
    }
    const u64 *words = reinterpret_cast<const u64 *>(surv);
    if (n <= CO_P_DIRECT) {
        if (blockIdx.x != 0) return;
        for (u32 i = threadIdx.x; i < 3 * n; i += CO_THREADS) reinterpret_cast<u64 *>(sv)[i] = __ldcg(words + i);
        __syncthreads();
        pareto_small(sv, n, flags, lim, idx_out, count_out);
        return;
    }
    // Many: the survivors are judged by all warps, against chunks of the list staged in shared memory;
    // those nobody rules out go to a second list.
    const u32 flat_warp = warp * gridDim.x + blockIdx.x;
    for (u32 g0 = 0; g0 < n; g0 += total_warps) {
        const u32 g = g0 + flat_warp;
        u64 mx = 0, my = 0, mi = 0;
        if (g < n) { mx = __ldcg(words + 3 * (size_t)g); my = __ldcg(words + 3 * (size_t)g + 1); mi = __ldcg(words + 3 * (size_t)g + 2); }
        bool out = g >= n;
        for (u32 c0 = 0; c0 < n; c0 += CO_P_CHUNK) {
            const u32 nc = min(CO_P_CHUNK, n - c0);
            __syncthreads();
            for (u32 i = threadIdx.x; i < 3 * nc; i += CO_THREADS) reinterpret_cast<u64 *>(sv)[i] = __ldcg(words + 3 * (size_t)c0 + i);
            __syncthreads();
            for (u32 i = lane; i < nc && !out; i += 32) {
                const P3 o = sv[i];
                out = dominates(o.x, o.y, mx, my) || (o.x == mx && o.y == my && o.idx < mi);
            }
        }
        if (!__any_sync(0xFFFFFFFFu, out) && lane == 0) {
            const u32 pos = atomicAdd(header + PH_FRONT, 1);                // pos < n <= PA_SURV_CAP
            front_list[pos].key = mx; front_list[pos].idx = mi;
        }
    }
    grid_barrier();
    // a front point's place is its rank in x
    const u32 nfr = __ldcg(header + PH_FRONT);
    const ulonglong2 *f = reinterpret_cast<const ulonglong2 *>(front_list);
    for (u32 g = flat_warp; g < nfr; g += total_warps) {
        const ulonglong2 me = __ldcg(f + g);
        u32 ahead = 0;
        for (u32 i = lane; i < nfr; i += 32) ahead += __ldcg(f + i).x < me.x ? 1u : 0u;
        ahead = __reduce_add_sync(0xFFFFFFFFu, ahead);
        if (lane == 0 && ahead < lim) idx_out[ahead] = me.y;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *count_out = nfr > GUIDE_PARETO_MAX ? 0xFFFFFFFFu : nfr;
}

// ---- host side -----------------------------------------------------------------------------------------

// The arrays a call touches, each once: metric(s) first, then the bounded ones not yet listed.
static int collect_arrays(const guide_outputs &o, const guide_constraints &c, int m0, int m1, Arr *arr) {
    int n = 0;
    auto add_metric = [&](int key) { arr[n++] = Arr{metric_array_of(o, key), 0.0, 0, key == GUIDE_THROUGHPUT ? 1 : 0}; };
    add_metric(m0);
    if (m1 >= 0) add_metric(m1);
    auto add_bound = [&](const double *p, double bound, int cmp) {
        for (int i = 0; i < n; i++)
            if (arr[i].p == p && arr[i].cmp == 0) { arr[i].bound = bound; arr[i].cmp = cmp; return; }
        arr[n++] = Arr{p, bound, cmp, 0};
    };
    if (c.max_ttft < INFINITY)
        add_bound(c.ttft_stat == GUIDE_STAT_MEAN ? o.ttft : c.ttft_stat == GUIDE_STAT_P50 ? o.ttft_p50 : o.ttft_p99, c.max_ttft, 1);
    if (c.max_latency < INFINITY) add_bound(o.latency, c.max_latency, 1);
    if (c.max_cost_per_hr < INFINITY) add_bound(o.cost_per_hr, c.max_cost_per_hr, 1);
    if (c.min_throughput > 0.0) add_bound(o.thr_decode, c.min_throughput, 2);
    return n;
}

// Does the device launch cooperatively, with CO_BLOCKS_PER_SM blocks resident per SM?  Asked once per device.
bool coop_select_ok() {
    static std::atomic<int> cached[64] = {};         // 0 unknown, 1 yes, 2 no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (!cached[dev]) {
        int coop = 0, t = 0, p = 0;
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t, k_topk_coop<MAX_ARR - 1, false>, CO_THREADS, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, k_pareto_coop<MAX_ARR, false>, CO_THREADS, 0);
        cached[dev] = (coop && !coop_disabled() && t >= (int)CO_BLOCKS_PER_SM && p >= (int)CO_BLOCKS_PER_SM) ? 1 : 2;
    }
    return cached[dev] == 1;
}

// A range one block can hold in its registers is one block; up to what CO_BLOCKS_PER_SM blocks per SM hold, a row per
// warp while that fills the machine.  Beyond, one block per SM: its pass over everything has enough in flight, and two
// selections on two streams fit side by side.
static u32 coop_grid(u64 n_rows) {
    if (n_rows <= CO_ONE_BLOCK_ROWS) return 1;
    const u64 full = std::min<u64>((u64)num_sms() * CO_BLOCKS_PER_SM, CO_MAX_BLOCKS);
    if (n_rows > full * CO_WARPS * CO_ROWS) return (u32)std::min<u64>((u64)num_sms(), CO_MAX_BLOCKS);
    return (u32)std::min<u64>((n_rows + CO_WARPS - 1) / CO_WARPS, full);
}

// All rows while the warps' registers hold them, else one out of every r, as many as they hold.
static Walk make_walk(u64 n_rows, u32 grid) {
    const u64 room = (u64)grid * CO_WARPS * CO_ROWS;
    Walk w;
    w.n_rows = n_rows;
    w.r = (u32)std::max<u64>((n_rows + room - 1) / room, 1);
    w.n_slots = n_rows / w.r;
    return w;
}

template <class... KArgs, class... Args>
static int launch_coop(void (*kernel)(KArgs...), u32 grid, cudaStream_t st, Args... args) {
    if (grid > 1) return launch_cooperative(kernel, grid, CO_THREADS, st, args...);
    GUIDE_CUDA(launch_dependent(kernel, 1, CO_THREADS, 0, st, args...));
    return GUIDE_OK;
}

// workspace region of a top-k call: KI minima[CO_BOUND_LIST] | KI spairs[CO_BOUND_LIST] | KI cand[TK_CAND_CAP]
size_t topk_coop_bytes() { return ((size_t)2 * CO_BOUND_LIST + TK_CAND_CAP) * sizeof(KI); }
// ... and of a Pareto call: P2 local[CO_DIRS][CO_MAX_BLOCKS] | P3 surv[PA_SURV_CAP] | P3 kept[PA_SURV_CAP] |
// KI front[PA_SURV_CAP] | u64 steps[CO_STEPS]
static constexpr size_t PC_SURV = (size_t)CO_DIRS * CO_MAX_BLOCKS * sizeof(P2), PC_KEPT = PC_SURV + (size_t)PA_SURV_CAP * sizeof(P3),
                        PC_FRONT = PC_KEPT + (size_t)PA_SURV_CAP * sizeof(P3), PC_STEPS = PC_FRONT + (size_t)PA_SURV_CAP * sizeof(KI);
size_t pareto_coop_bytes() { return PC_STEPS + CO_STEPS * sizeof(u64); }

template <int NA>
static CoopSrc<NA> coop_src(const Arr *arr, const guide_outputs &mat) {
    CoopSrc<NA> s;
    for (int i = 0; i < NA; i++) {
        s.a[i] = arr[i];
        s.free[i] = arr[i].cmp == 0;
        s.flip[i] = arr[i].cmp == 2 ? 0x80000000u : 0u;
        s.bnd[i] = arr[i].cmp == 2 ? -arr[i].bound : arr[i].bound;
    }
    s.status = mat.status;
    s.vec = mat_vec_ok(mat) ? ((uintptr_t)mat.status % 16 == 0 ? 2 : 1) : 0;
    return s;
}

template <int NA>
static int topk_coop_na(const Arr *arr, Range r, const guide_outputs &mat, u32 k, int negate, u32 *header, unsigned char *region,
                        u64 *idx_out, double *key_out, u32 *count_out, cudaStream_t st) {
    const CoopSrc<NA> s = coop_src<NA>(arr, mat);
    KI *minima = reinterpret_cast<KI *>(region), *spairs = minima + CO_BOUND_LIST, *cand = spairs + CO_BOUND_LIST;
    const u64 n_rows = (r.count + ROW - 1) / ROW;
    const u32 grid = coop_grid(n_rows);
    u32 group_log2 = 0;
    while (((grid * CO_WARPS) >> group_log2) > CO_BOUND_LIST) group_log2++;
    const Walk w = make_walk(n_rows, grid);
    return launch_coop(w.r == 1 ? k_topk_coop<NA, true> : k_topk_coop<NA, false>, grid, st, s, r, w, k, group_log2, header, minima, spairs, cand, negate,
                           idx_out, key_out, count_out);
}

int launch_topk_coop(Range r, const guide_outputs &mat, const guide_constraints &c, int key, u32 k, u32 *header,
                     unsigned char *region, u64 *idx_out, double *key_out, u32 *count_out, cudaStream_t st) {
    Arr arr[MAX_ARR];
    const int na = collect_arrays(mat, c, key, -1, arr);
    const int negate = key == GUIDE_THROUGHPUT;
    switch (na) {
    case 1: return topk_coop_na<1>(arr, r, mat, k, negate, header, region, idx_out, key_out, count_out, st);
    case 2: return topk_coop_na<2>(arr, r, mat, k, negate, header, region, idx_out, key_out, count_out, st);
    case 3: return topk_coop_na<3>(arr, r, mat, k, negate, header, region, idx_out, key_out, count_out, st);
    case 4: return topk_coop_na<4>(arr, r, mat, k, negate, header, region, idx_out, key_out, count_out, st);
    case 5: return topk_coop_na<5>(arr, r, mat, k, negate, header, region, idx_out, key_out, count_out, st);
    default: return fail(GUIDE_ERR_UNSUPPORTED, "a top-k call touches at most five arrays");
    }
}

template <int NA>
static int pareto_coop_na(const Arr *arr, Range r, const guide_outputs &mat, u32 *header, unsigned char *region, u64 *idx_out,
                          u32 cap, u32 *count_out, cudaStream_t st) {
    const CoopSrc<NA> s = coop_src<NA>(arr, mat);
    P2 *local = reinterpret_cast<P2 *>(region);
    P3 *surv = reinterpret_cast<P3 *>(region + PC_SURV), *kept = reinterpret_cast<P3 *>(region + PC_KEPT);
    KI *front = reinterpret_cast<KI *>(region + PC_FRONT);
    unsigned long long *steps = reinterpret_cast<unsigned long long *>(region + PC_STEPS);
    const u64 n_rows = (r.count + ROW - 1) / ROW;
    const u32 grid = coop_grid(n_rows);
    const Walk w = make_walk(n_rows, grid);
    return launch_coop(w.r == 1 ? k_pareto_coop<NA, true> : k_pareto_coop<NA, false>, grid, st, s, r, w, header, local, surv, kept, steps, front,
                           idx_out, cap, count_out);
}

int launch_pareto_coop(Range r, const guide_outputs &mat, const guide_constraints &c, int xm, int ym, u32 *header,
                       unsigned char *region, u64 *idx_out, u32 cap, u32 *count_out, cudaStream_t st) {
    Arr arr[MAX_ARR];
    const int na = collect_arrays(mat, c, xm, ym, arr);
    switch (na) {
    case 2: return pareto_coop_na<2>(arr, r, mat, header, region, idx_out, cap, count_out, st);
    case 3: return pareto_coop_na<3>(arr, r, mat, header, region, idx_out, cap, count_out, st);
    case 4: return pareto_coop_na<4>(arr, r, mat, header, region, idx_out, cap, count_out, st);
    case 5: return pareto_coop_na<5>(arr, r, mat, header, region, idx_out, cap, count_out, st);
    case 6: return pareto_coop_na<6>(arr, r, mat, header, region, idx_out, cap, count_out, st);
    default: return fail(GUIDE_ERR_UNSUPPORTED, "a Pareto call touches two to six arrays");
    }
}

}  // namespace guide

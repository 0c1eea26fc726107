// gj_factor.cu -- factor construction (Section 3.2, quantitative learning).
//
// A relation's potential is its exact frequency table: the distinct key
// tuples with their counts.  Here it is built by sorting the rows by their
// key tuple and cutting the sorted order into groups:
//
//   1. per key column, min and max (one read of every column);
//   2. each column becomes an unsigned field of ceil(log2(max-min+1)) bits,
//      packed into 64-bit words, most significant column first.  When the
//      key and the row id fit one word together, the row id rides in the low
//      bits and a keys-only LSD radix sort orders the key bits (a stable
//      sort of rows taken in row order keeps equal keys in row order);
//      otherwise (word, row id) pairs are sorted, word by word.  The first
//      pass builds the words from the key columns itself;
//   3. one group scan over the sorted words marks the rows whose key differs
//      from the previous row's, numbers these group heads (a single-pass
//      scan with decoupled lookback) and writes the row order, every group's
//      first position and key values, and the payload columns gathered
//      into group order.
//
// Sorted order is also the order the desummariser walks: groups sharing a
// separator value are contiguous (the separator columns lead the order) and
// inside a group rows keep increasing row id.
#include <algorithm>

#include "gj_factor_small.cuh"
#include "gj_lookback.cuh"
#include "gj_state.cuh"

namespace gj {
namespace {

constexpr int FT = 256;

struct ColSet {
    int ncol;
    const int32_t *col[MAX_KEYS];
};

__global__ void k_minmax_init(int nk, int32_t *mm) {
    int c = threadIdx.x;
    if (c < nk) { mm[2 * c] = INT32_MAX; mm[2 * c + 1] = INT32_MIN; }
}

// Range of column blockIdx.y: four 16-byte loads in flight per thread where the
// column is aligned, and one pair of atomics per block (a pair per warp queued
// up on the same two words: 1e7 rows x 2 columns 40 -> 22 us, three pairs of
// columns of 4e5 rows 63 -> 13).
__global__ void __launch_bounds__(FT) k_minmax(ColSet cs, int64_t n, int32_t *mm) {
    __shared__ int32_t s_lo[FT / 32], s_hi[FT / 32];
    const int c = blockIdx.y;
    const int32_t *col = cs.col[c];
    int32_t lo = INT32_MAX, hi = INT32_MIN;
    const int64_t stride = (int64_t)gridDim.x * FT;
    const int64_t at = (int64_t)blockIdx.x * FT + threadIdx.x;
    int64_t done = 0;
    if (((uintptr_t)col & 15) == 0) {
        const int64_t quads = n / 4;
        done = quads * 4;
        for (int64_t i = at; i < quads; i += 4 * stride) {
            int4 v[4];
#pragma unroll
            for (int u = 0; u < 4; u++) v[u] = __ldg((const int4 *)col + (i + u * stride < quads ? i + u * stride : i));
#pragma unroll
            for (int u = 0; u < 4; u++) {
                lo = min(lo, min(min(v[u].x, v[u].y), min(v[u].z, v[u].w)));
                hi = max(hi, max(max(v[u].x, v[u].y), max(v[u].z, v[u].w)));
            }
        }
    }
    for (int64_t i = done + at; i < n; i += stride) {
        const int32_t v = __ldg(col + i);
        lo = min(lo, v);
        hi = max(hi, v);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
        s_lo[threadIdx.x >> 5] = lo;
        s_hi[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < FT / 32; w++) {
            lo = min(lo, s_lo[w]);
            hi = max(hi, s_hi[w]);
        }
        if (lo <= hi) {
            atomicMin(&mm[2 * c], lo);
            atomicMax(&mm[2 * c + 1], hi);
        }
    }
}

// blocks per column: enough loads in flight, few enough atomics
inline unsigned minmax_blocks(Ctx &c, int64_t n, int cols) {
    const int64_t want = ceil_div(n, FT * 32), most = (int64_t)c.num_sms * 4 / cols;
    return (unsigned)std::max<int64_t>(1, std::min(want, most));
}

struct PackSpec {
    int ncol;
    const int32_t *col[MAX_KEYS];
    int32_t mn[MAX_KEYS];
    int shift[MAX_KEYS];
};

// keys[i] = packed fields of row (rows ? rows[i] : i); vals[i] = that row
__global__ void k_pack(PackSpec ps, const uint32_t *__restrict__ rows, int64_t n,
                       uint64_t *__restrict__ keys, uint32_t *__restrict__ vals) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT) {
        uint32_t r = rows ? rows[i] : (uint32_t)i;
        uint64_t k = 0;
#pragma unroll
        for (int c = 0; c < MAX_KEYS; c++) {
            if (c < ps.ncol && ps.shift[c] < 64)
                k |= (uint64_t)((uint32_t)ps.col[c][r] - (uint32_t)ps.mn[c]) << ps.shift[c];
        }
        keys[i] = k;
        vals[i] = r;
    }
}

// keys[i] = packed fields of row rows[i]; pos[i] = i (a position in the
// order rows[] lists the rows in)
__global__ void k_pack_pos(PackSpec ps, const uint32_t *__restrict__ rows, int64_t n,
                           uint64_t *__restrict__ keys, uint32_t *__restrict__ pos) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT) {
        const uint32_t r = rows[i];
        uint64_t k = 0;
#pragma unroll
        for (int c = 0; c < MAX_KEYS; c++) {
            if (c < ps.ncol && ps.shift[c] < 64)
                k |= (uint64_t)((uint32_t)ps.col[c][r] - (uint32_t)ps.mn[c]) << ps.shift[c];
        }
        keys[i] = k;
        pos[i] = (uint32_t)i;
    }
}

// the row ids and the low word in the final order: element i came from
// position pos[i] of the order the low word was sorted in
__global__ void k_compose(const uint32_t *__restrict__ pos, const uint32_t *__restrict__ perm0,
                          const uint64_t *__restrict__ lo0, int64_t n, uint32_t *__restrict__ perm,
                          uint64_t *__restrict__ lo) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT) {
        const uint32_t j = pos[i];
        perm[i] = perm0[j];
        lo[i] = lo0[j];
    }
}

// head[i] = i == 0 || key tuple of perm[i] != key tuple of perm[i-1]
__global__ void k_heads_packed(const uint64_t *__restrict__ keys, int64_t n, uint8_t *head) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT)
        head[i] = (i == 0) || keys[i] != keys[i - 1];
}

__global__ void k_heads_gather(ColSet cs, const uint32_t *__restrict__ perm, int64_t n,
                               uint8_t *head) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT) {
        uint8_t h = (i == 0);
        if (!h) {
            uint32_t a = perm[i], b = perm[i - 1];
            for (int c = 0; c < cs.ncol; c++)
                if (cs.col[c][a] != cs.col[c][b]) { h = 1; break; }
        }
        head[i] = h;
    }
}

__global__ void k_group_compact(ColSet cs, const uint32_t *__restrict__ perm,
                                const uint8_t *__restrict__ head, const uint32_t *__restrict__ gid,
                                int64_t n, int64_t G, uint32_t *gstart, int32_t *gkey) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT) {
        if (!head[i]) continue;
        uint32_t g = gid[i];
        gstart[g] = (uint32_t)i;
        uint32_t r = perm[i];
        for (int c = 0; c < cs.ncol; c++) gkey[(int64_t)c * G + g] = cs.col[c][r];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) gstart[G] = (uint32_t)n;
}

// Where each key column sits in the packed words of a sorted key (the low
// word, or the high one of a two-word key): value = ((word >> shift) &
// (2^bits - 1)) + min.  Columns outside the factor's order (projected
// away) are read through perm instead.
struct UnpackSpec {
    int ncol;
    int col[MAX_KEYS];
    int32_t mn[MAX_KEYS];
    int shift[MAX_KEYS];
    int bits[MAX_KEYS];
    int hi[MAX_KEYS];
    int nother;
    int other_col[MAX_KEYS];
    const int32_t *other[MAX_KEYS];
};

// sorted[c*n + i] = col_c[perm[i]]: the key columns in sorted order, one
// random read per column and row (used when the key spans several words)
__global__ void k_gather_cols(ColSet cs, const uint32_t *__restrict__ perm, int64_t n,
                              int32_t *__restrict__ sorted) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT) {
        uint32_t r = perm[i];
        for (int c = 0; c < cs.ncol; c++) sorted[(int64_t)c * n + i] = cs.col[c][r];
    }
}

// the columns a factor groups by (its order; all key columns unless some
// were projected away)
struct ColIdx {
    int n;
    int idx[MAX_KEYS];
};

__global__ void k_heads_sorted(const int32_t *__restrict__ sorted, ColIdx by, int64_t n, uint8_t *head) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT) {
        uint8_t h = (i == 0);
        for (int k = 0; k < by.n && !h; k++) {
            const int64_t c = by.idx[k];
            h = sorted[c * n + i] != sorted[c * n + i - 1];
        }
        head[i] = h;
    }
}

__global__ void k_group_compact_sorted(const int32_t *__restrict__ sorted, int nk,
                                       const uint8_t *__restrict__ head,
                                       const uint32_t *__restrict__ gid, int64_t n, int64_t G,
                                       uint32_t *gstart, int32_t *gkey) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT) {
        if (!head[i]) continue;
        uint32_t g = gid[i];
        gstart[g] = (uint32_t)i;
        for (int c = 0; c < nk; c++) gkey[(int64_t)c * G + g] = sorted[(int64_t)c * n + i];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) gstart[G] = (uint32_t)n;
}

template <class T>
__global__ void k_gather(const T *__restrict__ src, const uint32_t *__restrict__ perm, int64_t n,
                         T *__restrict__ dst) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT)
        dst[i] = src[perm[i]];
}

inline int grid_for(Ctx &c, int64_t n) {
    int64_t b = ceil_div(n, FT);
    int64_t cap = (int64_t)c.num_sms * 16;
    return (int)std::max<int64_t>(1, std::min(b, cap));
}

inline int bits_of(uint32_t range) { return range == 0 ? 0 : 32 - __builtin_clz(range); }

}  // namespace

void factor_free(Ctx &c, Factor &F) {
    dfree(c, F.perm);
    dfree(c, F.gstart);
    dfree(c, F.gkey);
    for (void *&p : F.pay) dfree(c, p);
    F.pay.clear();
}

namespace {

// ------------------------------------------------------------ group scan
// One pass over the sorted words: a row starts a group when its key differs
// from the previous row's; the groups are numbered by a single-pass scan
// with decoupled lookback, and the same pass writes the row order, every
// group's first position and key values, and the payloads in group order.
//   MODE 0  one word per row, the row id in its low row_bits bits
//   MODE 1  one word per row (the key), row order in perm_in
//   MODE 2  two words per row (hi, lo), row order in perm_in
constexpr int GS_THREADS = 256;
constexpr int GS_ITEMS = 16;
constexpr int GS_TILE = GS_THREADS * GS_ITEMS;

struct GroupScanSpec {
    const uint64_t *lo;           // sorted words (the low word of two)
    const uint64_t *hi;           // MODE 2: the high word
    const uint32_t *perm_in;      // MODE 1, 2
    uint32_t *perm_out;           // MODE 0: the row order taken from the words
    int row_bits;
    UnpackSpec u;                 // where each key column sits in the words
    int np;
    const void *pay_in[MAX_PAYLOADS];
    void *pay_out[MAX_PAYLOADS];
    int pw[MAX_PAYLOADS];
    uint32_t *gstart;             // [G+1]
    int32_t *gkey;                // column c of group g at c * gkey_stride + g
    int64_t gkey_stride;
    uint32_t *gcount;             // G
    unsigned long long *status;   // lookback state, one word per tile
    uint32_t *counter;            // tile counter
    uint32_t *err;
    uint32_t spin_limit;          // polls of a bounded wait
    int stall;                    // failure injection: tile 0 never publishes
};

// shared-memory slot of word q (q = 0 is the previous tile's last word): one
// pad word per 16, so that threads reading 16 consecutive words each are
// free of bank conflicts
__device__ __forceinline__ int gs_slot(int q) { return q + (q >> 4); }
constexpr int GS_SLOTS = GS_TILE + 1 + (GS_TILE + 1) / 16 + 1;

template <int MODE>
__global__ void __launch_bounds__(GS_THREADS, 4)
k_group_scan(GroupScanSpec s, int64_t n) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *s_lo = (uint64_t *)smem;
    uint64_t *s_hi = s_lo + GS_SLOTS;          // MODE 2 only
    __shared__ uint32_t s_wsum[GS_THREADS / 32];
    __shared__ uint32_t s_tile, s_carry;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_tile = atomicAdd(s.counter, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const int64_t base = (int64_t)tile * GS_TILE;
    if (base >= n) return;
    const int tile_n = (int)min((int64_t)GS_TILE, n - base);
    {
        // the tile's words, 16 loads in flight per thread
        uint64_t a[GS_ITEMS];
#pragma unroll
        for (int i = 0; i < GS_ITEMS; i++) {
            const int64_t idx = base + i * GS_THREADS + tid;
            a[i] = idx < n ? __ldg((const unsigned long long *)s.lo + idx) : 0ull;
        }
#pragma unroll
        for (int i = 0; i < GS_ITEMS; i++) s_lo[gs_slot(i * GS_THREADS + tid + 1)] = a[i];
        if (MODE == 2) {
#pragma unroll
            for (int i = 0; i < GS_ITEMS; i++) {
                const int64_t idx = base + i * GS_THREADS + tid;
                a[i] = idx < n ? __ldg((const unsigned long long *)s.hi + idx) : 0ull;
            }
#pragma unroll
            for (int i = 0; i < GS_ITEMS; i++) s_hi[gs_slot(i * GS_THREADS + tid + 1)] = a[i];
        }
    }
    if (tid == 0) {
        s_lo[0] = base > 0 ? s.lo[base - 1] : 0ull;
        if (MODE == 2) s_hi[0] = base > 0 ? s.hi[base - 1] : 0ull;
    }
    __syncthreads();
    // heads, row e = i * GS_THREADS + tid: one ballot per warp and i; the
    // tile's head counts per (i, warp) in row order, then their exclusive
    // prefix (warp 0, four entries a lane)
    __shared__ uint32_t s_cnt[GS_ITEMS * (GS_THREADS / 32)];
    __shared__ uint32_t s_hb[GS_ITEMS * (GS_THREADS / 32)];   // the ballots
    static_assert(GS_ITEMS * (GS_THREADS / 32) == 128, "four prefix entries per lane of warp 0");
#pragma unroll
    for (int i = 0; i < GS_ITEMS; i++) {
        const int e = i * GS_THREADS + tid;
        bool h = false;
        if (e < tile_n) {
            const uint64_t a = s_lo[gs_slot(e + 1)], b = s_lo[gs_slot(e)];
            if (MODE == 0) h = (a >> s.row_bits) != (b >> s.row_bits);
            else if (MODE == 1) h = a != b;
            else h = a != b || s_hi[gs_slot(e + 1)] != s_hi[gs_slot(e)];
            h = h || base + e == 0;
        }
        const uint32_t hb = __ballot_sync(0xffffffffu, h);
        if (lane == 0) {
            s_cnt[i * (GS_THREADS / 32) + warp] = __popc(hb);
            s_hb[i * (GS_THREADS / 32) + warp] = hb;
        }
    }
    __syncthreads();
    uint32_t agg = 0;
    if (warp == 0) {
        uint32_t v[4], sum = 0;
#pragma unroll
        for (int j = 0; j < 4; j++) { v[j] = s_cnt[lane * 4 + j]; sum += v[j]; }
        uint32_t x = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        agg = __shfl_sync(0xffffffffu, x, 31);
        uint32_t run = x - sum;
#pragma unroll
        for (int j = 0; j < 4; j++) { s_cnt[lane * 4 + j] = run; run += v[j]; }
        if (lane == 0) s_wsum[0] = agg;
    }
    __syncthreads();
    agg = s_wsum[0];
    // the tile's aggregate goes out first; the row order and the payloads do
    // not depend on the group numbering, so they are gathered while the
    // lookback waits on the predecessors
    // (published by the lane that later publishes the prefix: program order
    // keeps the prefix last)
    const bool silent = s.stall && tile == 0;
    if (warp == GS_THREADS / 32 - 1 && lane == 0 && !silent) publish_aggregate<uint32_t>(s.status, tile, agg);
    const uint64_t rmask = s.row_bits ? ((1ull << s.row_bits) - 1) : 0ull;
    // row order and payloads in group order, coalesced; each thread issues
    // its 16 gathers of a payload column together
    uint32_t r[GS_ITEMS];
#pragma unroll
    for (int i = 0; i < GS_ITEMS; i++) {
        const int e = i * GS_THREADS + tid;
        if (MODE == 0) r[i] = (uint32_t)(s_lo[gs_slot(e + 1)] & rmask);
        else r[i] = e < tile_n ? __ldg(s.perm_in + base + e) : 0u;
    }
    if (MODE == 0) {
#pragma unroll
        for (int i = 0; i < GS_ITEMS; i++) {
            const int e = i * GS_THREADS + tid;
            if (e < tile_n) s.perm_out[base + e] = r[i];
        }
    }
    for (int p = 0; p < s.np; p++) {
        if (s.pw[p] == 8) {
            const unsigned long long *src = (const unsigned long long *)s.pay_in[p];
            unsigned long long *dst = (unsigned long long *)s.pay_out[p];
            unsigned long long v[GS_ITEMS];
#pragma unroll
            for (int i = 0; i < GS_ITEMS; i++) v[i] = i * GS_THREADS + tid < tile_n ? __ldg(src + r[i]) : 0ull;
#pragma unroll
            for (int i = 0; i < GS_ITEMS; i++)
                if (i * GS_THREADS + tid < tile_n) dst[base + i * GS_THREADS + tid] = v[i];
        } else {
            const unsigned int *src = (const unsigned int *)s.pay_in[p];
            unsigned int *dst = (unsigned int *)s.pay_out[p];
            unsigned int v[GS_ITEMS];
#pragma unroll
            for (int i = 0; i < GS_ITEMS; i++) v[i] = i * GS_THREADS + tid < tile_n ? __ldg(src + r[i]) : 0u;
#pragma unroll
            for (int i = 0; i < GS_ITEMS; i++)
                if (i * GS_THREADS + tid < tile_n) dst[base + i * GS_THREADS + tid] = v[i];
        }
    }
    if (warp == GS_THREADS / 32 - 1) {
        const uint32_t carry = warp_lookback_published<uint32_t, AddU32>(s.status, tile, agg, lane, s.err,
                                                                          s.spin_limit);
        if (lane == 0) {
            s_carry = carry;
            if (base + GS_TILE >= n) {   // the last tile: the group count
                *s.gcount = carry + agg;
                s.gstart[carry + agg] = (uint32_t)n;
            }
        }
    }
    __syncthreads();
    // group starts and keys, row e = i * GS_THREADS + tid: the heads of one
    // (i, warp) take consecutive group numbers, so the stores of a warp are
    // contiguous where heads are dense
    const uint32_t carry = s_carry;
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll 1
    for (int i = 0; i < GS_ITEMS; i++) {
        const uint32_t hb = s_hb[i * (GS_THREADS / 32) + warp];
        if (!((hb >> lane) & 1u)) continue;
        const int e = i * GS_THREADS + tid;
        const int64_t idx = base + e;
        const uint32_t g = carry + s_cnt[i * (GS_THREADS / 32) + warp] + __popc(hb & lt);
        s.gstart[g] = (uint32_t)idx;
        const uint64_t klo = s_lo[gs_slot(e + 1)], khi = MODE == 2 ? s_hi[gs_slot(e + 1)] : 0ull;
        for (int c = 0; c < s.u.ncol; c++) {
            const uint64_t k = s.u.hi[c] ? khi : klo;
            const uint64_t mask = s.u.bits[c] >= 32 ? 0xFFFFFFFFull : ((1ull << s.u.bits[c]) - 1);
            const uint32_t v = (s.u.shift[c] < 64 ? (uint32_t)((k >> s.u.shift[c]) & mask) : 0u) + (uint32_t)s.u.mn[c];
            s.gkey[(int64_t)s.u.col[c] * s.gkey_stride + g] = (int32_t)v;
        }
        if (s.u.nother) {
            const uint32_t r = MODE == 0 ? (uint32_t)(klo & rmask) : s.perm_in[idx];
            for (int c = 0; c < s.u.nother; c++)
                s.gkey[(int64_t)s.u.other_col[c] * s.gkey_stride + g] = s.u.other[c][r];
        }
    }
}

// ------------------------------------------------------------ run groups
// A key that needs more than one word together with the row id: the rows are
// first sorted by the leading columns with the row id under them (keys-only).
// One kernel then orders every run of rows with equal leading columns by the
// remaining columns (ties stay in row order) and goes on to the groups: heads,
// group numbers (decoupled lookback), row order, group starts, keys and
// payloads.  A CTA owns the runs that start in its tile of RG_TILE rows and
// reads up to RUN_MAX rows past it for the last one.  A row's place in its run
// is the number of the run's rows before it, counted over the run staged in
// shared memory: rows of a run read the same words (broadcasts), and runs of
// any length share a warp, so short runs cost no idle lanes (a run per warp
// did: 1e7 runs of one or two rows took 4.9 ms).  The remaining columns are
// gathered by row id from one record per row that also holds the first
// payload column, so both cost one random sector.  Bound by those gathers
// (DRAM fetches 64 B for 16 useful ones).  Runs longer than RUN_MAX are not
// ordered here; a flag tells the host to build that factor the two-word way.
//
// Star of 1e7 rows x 4 keys of 20 bits (two columns lead, runs of ~1): run
// heads, their scan, the run sort and the group scan 5.4 ms -> 0.25 ms.
// 3e7 rows (one column leads, runs of ~30): 2.25 -> 1.00 ms; tiles of 2048 at
// 3 CTAs per SM 1.1 ms (fewer gathers in flight), two counting loops, before
// and after the row, 1.23 ms (their trip counts differ across a warp).  Runs of
// more than RG_LONG rows take three, cut at the row's word of 32, the same for
// the warp, and only the one over that word compares positions: the build of
// 2e7 rows in runs of 256 2.59 -> 1.86 ms (a bitonic network in registers, one
// warp per run: 2.03), of 200 2.31 -> 1.83 (2.18), of 100 1.66 -> 1.52 (1.94).
// From 32 rows on, 3e7 rows in runs of ~30 take 2.34 ms instead of 2.26.
constexpr int RUN_MAX = 256;
constexpr int RG_THREADS = 256;
constexpr int RG_TILE = 1280;
constexpr int RG_SPAN = RG_TILE + RUN_MAX;
constexpr int RG_ITEMS = RG_SPAN / RG_THREADS;
constexpr int RG_WORDS = RG_SPAN / 32;           // head bits of the span, 32 rows a word
constexpr int RG_TILE_WORDS = RG_TILE / 32;
constexpr int RG_LONG = 64;                      // rows of a run from which the counting splits by word
static_assert(RG_SPAN % RG_THREADS == 0 && RG_TILE % 32 == 0, "whole ballots");

struct RunGroupSpec {
    GroupScanSpec g;              // g.lo: lead << row_bits | row, sorted; u: rest is word 0, lead word 1
    const void *rec;              // [n] by row id: rest, or (rest, payload 0)
    uint32_t *too_long;           // set when a run exceeds RUN_MAX
};

template <bool PAY>
__global__ void __launch_bounds__(RG_THREADS, 5)
k_run_groups(RunGroupSpec rs, int64_t n) {
    const GroupScanSpec &s = rs.g;
    __shared__ uint64_t s_a[RG_SPAN + 1];          // row e of the span at e + 1; [0] the row before it
    __shared__ uint64_t s_r[RG_SPAN];
    __shared__ uint32_t s_hb[RG_WORDS];            // run heads, then group heads
    __shared__ int s_prev[RG_WORDS], s_next[RG_WORDS];   // last head before a word, first head after it
    __shared__ uint32_t s_cnt[RG_WORDS];
    __shared__ uint32_t s_tile, s_carry, s_agg;
    __shared__ int s_f, s_l;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_tile = atomicAdd(s.counter, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const int64_t base = (int64_t)tile * RG_TILE;
    if (base >= n) return;
    const int span = (int)min((int64_t)RG_SPAN, n - base);
    const uint64_t rmask = (1ull << s.row_bits) - 1;
    {
        uint64_t a[RG_ITEMS];
#pragma unroll
        for (int i = 0; i < RG_ITEMS; i++) {
            const int e = i * RG_THREADS + tid;
            a[i] = e < span ? __ldg((const unsigned long long *)s.lo + base + e) : 0ull;
        }
#pragma unroll
        for (int i = 0; i < RG_ITEMS; i++) s_a[i * RG_THREADS + tid + 1] = a[i];
        if (tid == 0) s_a[0] = base > 0 ? s.lo[base - 1] : 0ull;
    }
    __syncthreads();
    // run heads; positions past the last row count as heads (they end runs)
#pragma unroll
    for (int i = 0; i < RG_ITEMS; i++) {
        const int e = i * RG_THREADS + tid;
        const bool h = e >= span || base + e == 0 || (s_a[e + 1] >> s.row_bits) != (s_a[e] >> s.row_bits);
        const uint32_t hb = __ballot_sync(0xffffffffu, h);
        if (lane == 0) s_hb[e >> 5] = hb;
    }
    __syncthreads();
    // the nearest heads outside each word, as far as a run may reach
    if (tid < RG_WORDS) {
        int p = -1, q = RG_SPAN;
        for (int w = tid - 1; w >= 0 && w >= tid - RUN_MAX / 32 - 1; w--)
            if (s_hb[w]) { p = w * 32 + 31 - __clz((int)s_hb[w]); break; }
        for (int w = tid + 1; w < RG_WORDS && w <= tid + RUN_MAX / 32 + 1; w++)
            if (s_hb[w]) { q = w * 32 + __ffs((int)s_hb[w]) - 1; break; }
        s_prev[tid] = p;
        s_next[tid] = q;
    }
    if (warp == RG_THREADS / 32 - 1) {
        // the rows owned: from the tile's first head to the next tile's
        int f = RG_SPAN, l = RG_SPAN;
        for (int w = lane; w < RG_WORDS; w += 32) {
            if (!s_hb[w]) continue;
            const int e = w * 32 + __ffs((int)s_hb[w]) - 1;
            if (w < RG_TILE_WORDS) f = min(f, e); else l = min(l, e);
        }
        f = __reduce_min_sync(0xffffffffu, f);
        l = __reduce_min_sync(0xffffffffu, l);
        if (lane == 0) {
            // a run that starts before the tile or ends past the span is too
            // long; what is left stays in bounds and is thrown away
            const bool lost = f >= RG_TILE || (l >= RG_SPAN && base + RG_SPAN < n);
            s_f = min(f, span);
            s_l = f >= RG_TILE ? min(f, span) : min(l, span);
            if (lost && f < span) atomicOr(rs.too_long, 1u);
        }
    }
    __syncthreads();
    const int f = s_f, l = s_l;
    // the remaining columns (and the first payload) of the owned rows
    uint64_t r[RG_ITEMS], v[RG_ITEMS];
#pragma unroll
    for (int i = 0; i < RG_ITEMS; i++) {
        const int e = i * RG_THREADS + tid;
        const uint32_t row = (uint32_t)(s_a[e + 1] & rmask);
        r[i] = 0;
        v[i] = 0;
        if (e >= f && e < l) {
            if (PAY) {
                const ulonglong2 x = __ldg((const ulonglong2 *)rs.rec + row);
                r[i] = x.x;
                v[i] = x.y;
            } else {
                r[i] = __ldg((const unsigned long long *)rs.rec + row);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < RG_ITEMS; i++) s_r[i * RG_THREADS + tid] = r[i];
    __syncthreads();
    // a row's place: the rows of its run with a smaller rest, and those with
    // an equal one that come before it
    int pos[RG_ITEMS];
    bool over = false;
#pragma unroll
    for (int i = 0; i < RG_ITEMS; i++) {
        const int e = i * RG_THREADS + tid;
        pos[i] = e;
        if (e < f || e >= l) continue;
        const uint32_t hb = s_hb[e >> 5];
        const uint32_t le = hb & (0xffffffffu >> (31 - lane)), gt = lane == 31 ? 0u : hb & (0xffffffffu << (lane + 1));
        const int b0 = le ? (e & ~31) + 31 - __clz((int)le) : s_prev[e >> 5];
        const int b1 = min(gt ? (e & ~31) + __ffs((int)gt) - 1 : s_next[e >> 5], l);
        if (b0 < f || b1 - b0 > RUN_MAX) { over = true; continue; }
        const uint64_t x = r[i];
        int k = b0, j = b0, end = b1;
        if (b1 - b0 > RG_LONG) {
            // rows before this one's word come first if they are equal
            for (; j < (e & ~31); j++) k += s_r[j] <= x ? 1 : 0;
            end = min(b1, (e & ~31) + 32);
        }
#pragma unroll 4
        for (; j < end; j++) {
            const uint64_t y = s_r[j];
            k += (y < x || (y == x && j < e)) ? 1 : 0;
        }
        for (; j < b1; j++) k += s_r[j] < x ? 1 : 0;
        pos[i] = k;
    }
    if (over) atomicOr(rs.too_long, 1u);
    uint64_t a[RG_ITEMS];
#pragma unroll
    for (int i = 0; i < RG_ITEMS; i++) a[i] = s_a[i * RG_THREADS + tid + 1];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RG_ITEMS; i++) {
        const int e = i * RG_THREADS + tid;
        if (e < f || e >= l) continue;
        s_a[pos[i] + 1] = a[i];
        s_r[pos[i]] = r[i];
        s.perm_out[base + pos[i]] = (uint32_t)(a[i] & rmask);
        if (PAY) {
            if (s.pw[0] == 8) ((unsigned long long *)s.pay_out[0])[base + pos[i]] = v[i];
            else ((unsigned int *)s.pay_out[0])[base + pos[i]] = (unsigned int)v[i];
        }
    }
    __syncthreads();
    // group heads of the ordered rows
#pragma unroll
    for (int i = 0; i < RG_ITEMS; i++) {
        const int e = i * RG_THREADS + tid;
        const bool h = e >= f && e < l && (e == f || s_r[e] != s_r[e - 1] ||
                                           (s_a[e + 1] >> s.row_bits) != (s_a[e] >> s.row_bits));
        const uint32_t hb = __ballot_sync(0xffffffffu, h);
        if (lane == 0) s_hb[e >> 5] = hb;
    }
    __syncthreads();
    const bool silent = s.stall && tile == 0;
    if (warp == 0) {
        uint32_t run = 0;
#pragma unroll
        for (int w0 = 0; w0 < RG_WORDS; w0 += 32) {
            const int w = w0 + lane;
            const uint32_t c = w < RG_WORDS ? __popc(s_hb[w]) : 0u;
            uint32_t x = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
                if (lane >= d) x += y;
            }
            if (w < RG_WORDS) s_cnt[w] = run + x - c;
            run += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0 && !silent) publish_aggregate<uint32_t>(s.status, tile, run);
        const uint32_t carry = warp_lookback_published<uint32_t, AddU32>(s.status, tile, run, lane, s.err,
                                                                          s.spin_limit);
        if (lane == 0) {
            s_carry = carry;
            if (base + RG_TILE >= n) {   // the last tile: the group count
                *s.gcount = carry + run;
                s.gstart[carry + run] = (uint32_t)n;
            }
        }
    } else {
        // payloads outside the record, gathered meanwhile
        for (int p = PAY ? 1 : 0; p < s.np; p++)
            for (int e = tid - 32; e < l; e += RG_THREADS - 32) {
                if (e < f) continue;
                const uint32_t row = (uint32_t)(s_a[e + 1] & rmask);
                if (s.pw[p] == 8)
                    ((unsigned long long *)s.pay_out[p])[base + e] = __ldg((const unsigned long long *)s.pay_in[p] + row);
                else
                    ((unsigned int *)s.pay_out[p])[base + e] = __ldg((const unsigned int *)s.pay_in[p] + row);
            }
    }
    __syncthreads();
    const uint32_t carry = s_carry;
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll 1
    for (int i = 0; i < RG_ITEMS; i++) {
        const int e = i * RG_THREADS + tid;
        const uint32_t hb = s_hb[e >> 5];
        if (!((hb >> lane) & 1u)) continue;
        const uint32_t g = carry + s_cnt[e >> 5] + __popc(hb & lt);
        s.gstart[g] = (uint32_t)(base + e);
        const uint64_t kr = s_r[e], kl = s_a[e + 1] >> s.row_bits;
        for (int c = 0; c < s.u.ncol; c++) {
            const uint64_t k = s.u.hi[c] ? kl : kr;
            const uint64_t mask = s.u.bits[c] >= 32 ? 0xFFFFFFFFull : ((1ull << s.u.bits[c]) - 1);
            const uint32_t x = (s.u.shift[c] < 64 ? (uint32_t)((k >> s.u.shift[c]) & mask) : 0u) + (uint32_t)s.u.mn[c];
            s.gkey[(int64_t)s.u.col[c] * s.gkey_stride + g] = (int32_t)x;
        }
        for (int c = 0; c < s.u.nother; c++)
            s.gkey[(int64_t)s.u.other_col[c] * s.gkey_stride + g] = s.u.other[c][(uint32_t)(s_a[e + 1] & rmask)];
    }
}

// one record per row, in row order (sequential reads): the remaining columns
// packed into a word, and with PAY the first payload column
template <bool PAY>
__global__ void k_pack_rest(PackSrc ps, const void *pay, int pw, int64_t n, void *__restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT) {
        const unsigned long long w = pack_word(ps, i);
        if (PAY) {
            const unsigned long long v = pw == 8 ? __ldg((const unsigned long long *)pay + i)
                                                 : (unsigned long long)__ldg((const unsigned int *)pay + i);
            ((ulonglong2 *)out)[i] = make_ulonglong2(w, v);
        } else {
            ((unsigned long long *)out)[i] = w;
        }
    }
}

// One factor build in two stages, so that the builds of several relations
// share their host synchronisations: the key ranges (for the packed field
// widths) before the sort, and the group counts (for the group arrays)
// after it.
struct FactorBuild {
    Relation *R = nullptr;
    Factor *F = nullptr;
    std::vector<int> bits;
    std::vector<std::vector<int>> words;
    // fused path (keys of at most two words): the group scan wrote gstart,
    // the keys at stride n, the payloads and the count
    bool fused = false;
    uint32_t *gstart = nullptr;    // [n+1]
    int32_t *gkey_n = nullptr;     // [nk*n]
    uint32_t *gcount = nullptr;
    // wide keys sorted by their leading columns, then run by run
    bool force_two = false;        // build the two-word way (a run was too long)
    uint32_t *too_long = nullptr;
    // keys of more than two words
    uint8_t *head = nullptr;
    uint32_t *gid = nullptr;
    int32_t *sorted = nullptr;
};

void fb_free(Ctx &c, FactorBuild &b) {
    dfree(c, b.too_long);
    dfree(c, b.gstart);
    dfree(c, b.gkey_n);
    dfree(c, b.gcount);
    dfree(c, b.head);
    dfree(c, b.gid);
    dfree(c, b.sorted);
}

// the key fields of `order` for the group scan: column cols[i] at bit
// shift[i] of word hi[i]
UnpackSpec unpack_spec(const Relation &R, const std::vector<int> &order,
                       const std::vector<std::vector<int>> &words, const std::vector<int> &bits,
                       int row_bits) {
    UnpackSpec u{};
    for (size_t w = 0; w < words.size(); w++) {
        int shift = w == 0 ? row_bits : 0;
        for (int col : words[w]) {   // least significant first, as packed
            u.col[u.ncol] = col;
            u.mn[u.ncol] = R.kmin[col];
            u.shift[u.ncol] = shift;
            u.bits[u.ncol] = bits[col];
            u.hi[u.ncol] = (int)w;
            shift += bits[col];
            u.ncol++;
        }
    }
    for (int col = 0; col < R.nk; col++) {
        if (std::find(order.begin(), order.end(), col) != order.end()) continue;
        u.other_col[u.nother] = col;
        u.other[u.nother] = R.key[col];
        u.nother++;
    }
    return u;
}

PackSrc pack_src(const Relation &R, const std::vector<int> &wcols, const std::vector<int> &bits,
                 int row_bits) {
    PackSrc ps{};
    ps.ncol = (int)wcols.size();
    ps.row_bits = row_bits;
    int shift = row_bits;
    for (int i = 0; i < ps.ncol; i++) {   // wcols[0] is the least significant
        const int col = wcols[i];
        ps.col[i] = R.key[col];
        ps.mn[i] = R.kmin[col];
        ps.shift[i] = shift;
        shift += bits[col];
    }
    return ps;
}

// the lookback state of a group scan over `tiles` tiles (held by tmp)
cudaError_t scan_state(Ctx &c, Temps &tmp, GroupScanSpec &gs, int64_t tiles) {
    unsigned long long *state = nullptr;
    GJ_CUDA_TRY(tmp.alloc(&state, tiles + 2));
    GJ_CUDA_TRY(cudaMemsetAsync(state, 0, 8 * (tiles + 2), c.stream));
    gs.counter = (uint32_t *)state;
    gs.status = state + 2;
    gs.err = c.err;
    gs.spin_limit = c.spin_limit;
    gs.stall = c.test_stall ? 1 : 0;
    return cudaSuccess;
}

template <int MODE>
cudaError_t launch_group_scan(Ctx &c, GroupScanSpec &gs, int64_t n) {
    const int64_t tiles = ceil_div(n, GS_TILE);
    Temps tmp(c);
    GJ_CUDA_TRY(scan_state(c, tmp, gs, tiles));
    const size_t smem = (size_t)GS_SLOTS * 8 * (MODE == 2 ? 2 : 1);
    GJ_CUDA_TRY(cudaFuncSetAttribute(k_group_scan<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_group_scan<MODE><<<(unsigned)tiles, GS_THREADS, smem, c.stream>>>(gs, n); c.launches++;
    return cudaGetLastError();
}

// The leading columns of `order` that fit one word with the row id, when
// the remaining ones fit another: their number, else 0.
int run_split(const std::vector<int> &order, const std::vector<int> &bits, int row_bits) {
    int nlead = 0, used = row_bits;
    while (nlead < (int)order.size() && used + bits[order[nlead]] <= 64) used += bits[order[nlead++]];
    if (nlead == 0 || nlead == (int)order.size()) return 0;
    int rest = 0;
    for (size_t i = nlead; i < order.size(); i++) rest += bits[order[i]];
    return rest <= 64 ? nlead : 0;
}

// stage 1 (key ranges known): rows sorted by the key tuple; keys of one or
// two words go straight on to the group scan (the group count lands in
// b.gcount), longer keys mark and number their group heads
cudaError_t fb_sort(Ctx &c, FactorBuild &b) {
    Relation &R = *b.R;
    Factor &F = *b.F;
    const std::vector<int> &order = F.order;
    F.n = R.n;
    const int64_t n = R.n;
    if (n == 0) {
        GJ_CUDA_TRY(dalloc(c, &F.perm, 1));
        return cudaSuccess;
    }
    // field widths, least significant column last in `order`
    std::vector<int> &bits = b.bits;
    bits.assign(R.nk, 0);
    for (int i = 0; i < R.nk; i++)
        bits[i] = bits_of((uint32_t)((int64_t)R.kmax[i] - (int64_t)R.kmin[i]));
    int kbits = 0;
    for (int col : order) kbits += bits[col];
    const int row_bits = bits_of((uint32_t)(n - 1));
    // cut the order into words of <= 64 bits, starting from the least
    // significant column
    std::vector<std::vector<int>> &words = b.words;
    {
        std::vector<int> cur;
        int used = 0;
        for (int i = (int)order.size() - 1; i >= 0; i--) {
            int col = order[i];
            if (used + bits[col] > 64 && !cur.empty()) {
                words.push_back(cur);
                cur.clear();
                used = 0;
            }
            cur.push_back(col);
            used += bits[col];
        }
        if (!cur.empty()) words.push_back(cur);
    }
    if (words.size() <= 2) {
        // the fused path: sort, then one group scan
        b.fused = true;
        GroupScanSpec gs{};
        GJ_CUDA_TRY(dalloc(c, &b.gstart, n + 1));
        GJ_CUDA_TRY(dalloc(c, &b.gkey_n, (size_t)R.nk * n));
        GJ_CUDA_TRY(dalloc(c, &b.gcount, 1));
        for (int p = 0; p < R.np; p++) {
            void *d = nullptr;
            GJ_CUDA_TRY(dalloc_bytes(c, &d, (size_t)R.pw[p] * n));
            F.pay.push_back(d);
            gs.pay_in[p] = R.pay[p];
            gs.pay_out[p] = d;
            gs.pw[p] = R.pw[p];
        }
        gs.np = R.np;
        gs.gstart = b.gstart;
        gs.gkey = b.gkey_n;
        gs.gkey_stride = n;
        gs.gcount = b.gcount;
        // temporaries of this build, freed on every way out
        Temps tmp(c);
        uint64_t *k1 = nullptr, *k2 = nullptr, *kres = nullptr;
        GJ_CUDA_TRY(tmp.alloc(&k1, n));
        GJ_CUDA_TRY(tmp.alloc(&k2, n));
        if (words.size() == 1 && kbits + row_bits <= 64) {
            // MODE 0: the row id rides under the key; a keys-only sort of the
            // key bits
            PackSrc ps = pack_src(R, words[0], bits, row_bits);
            GJ_CUDA_TRY(radix_sort_words(c, &ps, k1, k2, nullptr, nullptr, n, row_bits, kbits, &kres, nullptr));
            GJ_CUDA_TRY(dalloc(c, &F.perm, n));
            gs.lo = kres;
            gs.perm_out = F.perm;
            gs.row_bits = row_bits;
            gs.u = unpack_spec(R, order, words, bits, row_bits);
            GJ_CUDA_TRY(launch_group_scan<0>(c, gs, n));
        } else if (words.size() == 1) {
            // MODE 1: (key, row id) pairs
            uint32_t *v1 = nullptr, *v2 = nullptr, *vres = nullptr;
            GJ_CUDA_TRY(tmp.alloc(&v1, n));
            GJ_CUDA_TRY(tmp.alloc(&v2, n));
            PackSrc ps = pack_src(R, words[0], bits, 0);
            GJ_CUDA_TRY(radix_sort_words(c, &ps, k1, k2, v1, v2, n, 0, kbits, &kres, &vres));
            // the sorted row ids become the factor's row order
            F.perm = vres;
            tmp.keep(vres);
            gs.lo = kres;
            gs.perm_in = F.perm;
            gs.u = unpack_spec(R, order, words, bits, 0);
            GJ_CUDA_TRY(launch_group_scan<1>(c, gs, n));
        } else if (int nlead = run_split(order, bits, row_bits); !b.force_two && nlead > 0) {
            // the leading columns with the row id under them (keys-only);
            // then each run of equal leading columns ordered by the rest and
            // cut into groups in one kernel
            std::vector<int> lead(order.begin(), order.begin() + nlead);
            std::vector<int> rest(order.begin() + nlead, order.end());
            std::reverse(lead.begin(), lead.end());   // least significant first
            std::reverse(rest.begin(), rest.end());
            int lead_bits = 0;
            for (int col : lead) lead_bits += bits[col];
            PackSrc pa = pack_src(R, lead, bits, row_bits);
            GJ_CUDA_TRY(radix_sort_words(c, &pa, k1, k2, nullptr, nullptr, n, row_bits, lead_bits, &kres, nullptr));
            GJ_CUDA_TRY(dalloc(c, &F.perm, n));
            GJ_CUDA_TRY(dalloc(c, &b.too_long, 1));
            GJ_CUDA_TRY(cudaMemsetAsync(b.too_long, 0, 4, c.stream));
            const bool pay = R.np > 0;
            void *rec = nullptr;
            GJ_CUDA_TRY(tmp.alloc_bytes(&rec, (size_t)(pay ? 16 : 8) * n));
            const PackSrc pr = pack_src(R, rest, bits, 0);
            if (pay) k_pack_rest<true><<<grid_for(c, n), FT, 0, c.stream>>>(pr, R.pay[0], R.pw[0], n, rec);
            else k_pack_rest<false><<<grid_for(c, n), FT, 0, c.stream>>>(pr, nullptr, 0, n, rec);
            c.launches++;
            GJ_CUDA_TRY(cudaGetLastError());
            gs.lo = kres;
            gs.perm_out = F.perm;
            gs.row_bits = row_bits;
            gs.u = unpack_spec(R, order, {rest, lead}, bits, 0);
            RunGroupSpec rg{};
            rg.rec = rec;
            rg.too_long = b.too_long;
            const int64_t tiles = ceil_div(n, RG_TILE);
            GJ_CUDA_TRY(scan_state(c, tmp, gs, tiles));
            rg.g = gs;
            if (pay) k_run_groups<true><<<(unsigned)tiles, RG_THREADS, 0, c.stream>>>(rg, n);
            else k_run_groups<false><<<(unsigned)tiles, RG_THREADS, 0, c.stream>>>(rg, n);
            c.launches++;
            GJ_CUDA_TRY(cudaGetLastError());
        } else {
            // MODE 2: the low word sorts with row ids; the high word sorts
            // carrying positions in the low word's order, and one gather then
            // brings the row ids and the low word into the final order
            uint32_t *v1 = nullptr, *v2 = nullptr, *perm0 = nullptr;
            GJ_CUDA_TRY(tmp.alloc(&v1, n));
            GJ_CUDA_TRY(tmp.alloc(&v2, n));
            PackSrc ps = pack_src(R, words[0], bits, 0);
            int lo_bits = 0;
            for (int col : words[0]) lo_bits += bits[col];
            uint64_t *lo_sorted = nullptr;
            GJ_CUDA_TRY(radix_sort_words(c, &ps, k1, k2, v1, v2, n, 0, lo_bits, &lo_sorted, &perm0));
            uint32_t *vfree = perm0 == v1 ? v2 : v1;   // free buffer of n values
            uint64_t *kfree = lo_sorted == k1 ? k2 : k1;
            PackSpec ph{};
            ph.ncol = (int)words[1].size();
            int shift = 0;
            for (int i = 0; i < ph.ncol; i++) {
                const int col = words[1][i];
                ph.col[i] = R.key[col];
                ph.mn[i] = R.kmin[col];
                ph.shift[i] = shift;
                shift += bits[col];
            }
            uint64_t *h1 = nullptr, *hres = nullptr;
            uint32_t *pos2 = nullptr, *pres = nullptr;
            GJ_CUDA_TRY(tmp.alloc(&h1, n));
            GJ_CUDA_TRY(tmp.alloc(&pos2, n));
            k_pack_pos<<<grid_for(c, n), FT, 0, c.stream>>>(ph, perm0, n, kfree, vfree); c.launches++;
            GJ_CUDA_TRY(cudaGetLastError());
            GJ_CUDA_TRY(radix_sort_words(c, nullptr, kfree, h1, vfree, pos2, n, 0, shift, &hres, &pres));
            uint64_t *lo_final = hres == kfree ? h1 : kfree;   // the buffer hres does not hold
            uint32_t *perm = pres == vfree ? pos2 : vfree;
            k_compose<<<grid_for(c, n), FT, 0, c.stream>>>(pres, perm0, lo_sorted, n, perm, lo_final); c.launches++;
            GJ_CUDA_TRY(cudaGetLastError());
            F.perm = perm;
            tmp.keep(perm);
            gs.lo = lo_final;
            gs.hi = hres;
            gs.perm_in = F.perm;
            gs.u = unpack_spec(R, order, words, bits, 0);
            GJ_CUDA_TRY(launch_group_scan<2>(c, gs, n));
        }
        return cudaSuccess;
    }
    // keys of three or more words: (word, row id) sorts word by word, then
    // the key columns are brought into sorted order once and the groups are
    // found with sequential reads
    GJ_CUDA_TRY(dalloc(c, &F.perm, n));
    uint64_t *keys = nullptr;
    Temps tmp(c);
    GJ_CUDA_TRY(tmp.alloc(&keys, n));
    for (size_t w = 0; w < words.size(); w++) {   // least significant word first
        const std::vector<int> &wcols = words[w];
        PackSpec ps{};
        ps.ncol = (int)wcols.size();
        int shift = 0;
        for (int i = 0; i < ps.ncol; i++) {   // wcols[0] is the least significant
            int col = wcols[i];
            ps.col[i] = R.key[col];
            ps.mn[i] = R.kmin[col];
            ps.shift[i] = shift;
            shift += bits[col];
        }
        k_pack<<<grid_for(c, n), FT, 0, c.stream>>>(ps, w == 0 ? nullptr : F.perm, n, keys, F.perm); c.launches++;
        GJ_CUDA_TRY(cudaGetLastError());
        GJ_CUDA_TRY(radix_sort_u64_u32(c, keys, F.perm, n, shift));
    }
    tmp.free(keys);
    GJ_CUDA_TRY(dalloc(c, &b.head, n));
    GJ_CUDA_TRY(dalloc(c, &b.gid, n));
    GJ_CUDA_TRY(dalloc(c, &b.gcount, 1));
    ColSet all{};
    all.ncol = R.nk;
    for (int i = 0; i < R.nk; i++) all.col[i] = R.key[i];
    GJ_CUDA_TRY(dalloc(c, &b.sorted, (size_t)R.nk * n));
    k_gather_cols<<<grid_for(c, n), FT, 0, c.stream>>>(all, F.perm, n, b.sorted); c.launches++;
    ColIdx by{};
    by.n = (int)order.size();
    for (int i = 0; i < by.n; i++) by.idx[i] = order[i];
    k_heads_sorted<<<grid_for(c, n), FT, 0, c.stream>>>(b.sorted, by, n, b.head); c.launches++;
    GJ_CUDA_TRY(cudaGetLastError());
    GJ_CUDA_TRY(scan_u32(c, nullptr, b.head, b.gid, n, b.gcount));
    return cudaSuccess;
}

// stage 2 (group count G known): the group arrays at their final size,
// payloads in group order; frees the stage's temporaries
cudaError_t fb_groups(Ctx &c, FactorBuild &b, int64_t G) {
    Relation &R = *b.R;
    Factor &F = *b.F;
    const int64_t n = R.n;
    if (n == 0) {
        F.G = 0;
        GJ_CUDA_TRY(dalloc(c, &F.gstart, 1));
        GJ_CUDA_TRY(cudaMemsetAsync(F.gstart, 0, sizeof(uint32_t), c.stream));
        GJ_CUDA_TRY(dalloc(c, &F.gkey, 1));
        for (int p = 0; p < R.np; p++) {
            void *d = nullptr;
            GJ_CUDA_TRY(dalloc_bytes(c, &d, 16));
            F.pay.push_back(d);
        }
        return cudaSuccess;
    }
    F.G = G;
    if (b.fused) {
        // group starts stay in their n + 1 slots, and the keys in their
        // columns of n where at least half the rows are groups of their own
        // (moving 3e7 x 4 keys took 0.15 ms and another 0.5 GB); fewer groups
        // move to columns of G, so that a factor keeps no more than twice its
        // keys
        F.gstart = b.gstart;
        b.gstart = nullptr;
        if (2 * G >= n) {
            F.gkey = b.gkey_n;
            F.kstride = n;
            b.gkey_n = nullptr;
        } else {
            GJ_CUDA_TRY(dalloc(c, &F.gkey, (size_t)R.nk * G));
            F.kstride = G;
            CopySet cs;
            for (int k = 0; k < R.nk; k++) cs.add(F.key(k), b.gkey_n + (int64_t)k * n, 4 * G);
            if (cs.n) GJ_CUDA_TRY(copy_arrays(c, cs));
        }
        fb_free(c, b);
        return cudaSuccess;
    }
    GJ_CUDA_TRY(dalloc(c, &F.gstart, F.G + 1));
    GJ_CUDA_TRY(dalloc(c, &F.gkey, (size_t)R.nk * F.G));
    F.kstride = F.G;
    k_group_compact_sorted<<<grid_for(c, n), FT, 0, c.stream>>>(b.sorted, R.nk, b.head, b.gid, n, F.G,
                                                                F.gstart, F.gkey); c.launches++;
    GJ_CUDA_TRY(cudaGetLastError());
    for (int p = 0; p < R.np; p++) {
        void *d = nullptr;
        GJ_CUDA_TRY(dalloc_bytes(c, &d, (size_t)R.pw[p] * n));
        if (R.pw[p] == 8) {
            k_gather<uint64_t><<<grid_for(c, n), FT, 0, c.stream>>>(
                (const uint64_t *)R.pay[p], F.perm, n, (uint64_t *)d); c.launches++;
        } else {
            k_gather<uint32_t><<<grid_for(c, n), FT, 0, c.stream>>>(
                (const uint32_t *)R.pay[p], F.perm, n, (uint32_t *)d); c.launches++;
        }
        GJ_CUDA_TRY(cudaGetLastError());
        F.pay.push_back(d);
    }
    fb_free(c, b);
    return cudaSuccess;
}

}  // namespace

// Builds the factors F[i] (order set) of relations R[i] together: the small
// ones in one launch, the others' missing key ranges, one readback of both,
// the others' sorts, one readback of their group counts, then the group arrays
// (their work has ended when the call returns).
// *err_word receives the device error word, read back with the last of these.
// On error the caller frees the factors (factor_free); temporaries are freed
// here.
cudaError_t factor_build_many(Ctx &c, const std::vector<Relation *> &R, const std::vector<Factor *> &F,
                              uint32_t *err_word) {
    const size_t m = R.size();
    *err_word = 0;
    if (m * (SF_OUT + 2 * MAX_KEYS) * 4 + 64 > (1 << 16)) return cudaErrorInvalidValue;
    auto read_err = [&](void *host) { return cudaMemcpyAsync(host, c.err, 4, cudaMemcpyDeviceToHost, c.stream); };
    std::vector<char> done(m, 0);
    Temps tmp(c);
    int32_t *words = nullptr;      // the small builds' reports, then the ranges
    std::vector<SmallFactor> small;
    std::vector<size_t> small_at;
    std::vector<Relation *> need;  // relations whose key ranges are to be found
    size_t n_words = 0;
    for (size_t i = 0; i < m; i++) {
        if (R[i]->n > 0 && R[i]->n <= SF_MAX && !c.test_stall) {
            small.push_back({R[i], F[i], nullptr});
            small_at.push_back(i);
            n_words += SF_OUT;
        } else if (!R[i]->have_minmax && std::find(need.begin(), need.end(), R[i]) == need.end()) {
            need.push_back(R[i]);
            n_words += 2 * R[i]->nk;
        }
    }
    if (n_words) {
        GJ_CUDA_TRY(tmp.alloc(&words, n_words));
        size_t off = 0;
        for (SmallFactor &f : small) {
            f.out = words + off;
            off += SF_OUT;
            GJ_CUDA_TRY(dalloc(c, &f.F->perm, f.R->n));
            GJ_CUDA_TRY(dalloc(c, &f.F->gstart, f.R->n + 1));
            GJ_CUDA_TRY(dalloc(c, &f.F->gkey, (size_t)f.R->nk * f.R->n));
            for (int p = 0; p < f.R->np; p++) {
                void *d = nullptr;
                GJ_CUDA_TRY(dalloc_bytes(c, &d, (size_t)f.R->pw[p] * f.R->n));
                f.F->pay.push_back(d);
            }
        }
        GJ_CUDA_TRY(small_factors(c, small));
        for (Relation *r : need) {
            if (r->n > 0) {
                ColSet cs{};
                cs.ncol = r->nk;
                for (int i = 0; i < r->nk; i++) cs.col[i] = r->key[i];
                k_minmax_init<<<1, 32, 0, c.stream>>>(r->nk, words + off); c.launches++;
                const dim3 grid(minmax_blocks(c, r->n, r->nk), r->nk);
                k_minmax<<<grid, FT, 0, c.stream>>>(cs, r->n, words + off); c.launches++;
                GJ_CUDA_TRY(cudaGetLastError());
            }
            off += 2 * r->nk;
        }
        // device->host readbacks go through the pinned buffer, then sync
        int32_t *h = (int32_t *)c.pinned;
        GJ_CUDA_TRY(cudaMemcpyAsync(h, words, sizeof(int32_t) * n_words, cudaMemcpyDeviceToHost, c.stream));
        GJ_CUDA_TRY(read_err(h + n_words));
        GJ_CUDA_TRY(cudaStreamSynchronize(c.stream));
        *err_word = (uint32_t)h[n_words];
        off = 0;
        for (size_t k = 0; k < small.size(); k++, off += SF_OUT) {
            const size_t i = small_at[k];
            Relation &r = *R[i];
            r.kmin.assign(r.nk, 0);
            r.kmax.assign(r.nk, 0);
            for (int x = 0; x < r.nk; x++) { r.kmin[x] = h[off + 2 + 2 * x]; r.kmax[x] = h[off + 3 + 2 * x]; }
            r.have_minmax = true;
            if (h[off + 1]) {
                F[i]->n = r.n;
                F[i]->G = h[off];
                F[i]->kstride = h[off];
                done[i] = 1;
            } else {
                factor_free(c, *F[i]);   // a wide key: built below
            }
        }
        for (Relation *r : need) {
            r->kmin.assign(r->nk, 0);
            r->kmax.assign(r->nk, 0);
            if (r->n > 0)
                for (int i = 0; i < r->nk; i++) { r->kmin[i] = h[off + 2 * i]; r->kmax[i] = h[off + 2 * i + 1]; }
            r->have_minmax = true;
            off += 2 * r->nk;
        }
        tmp.free(words);
    }
    std::vector<FactorBuild> b;
    for (size_t i = 0; i < m; i++) {
        if (done[i]) continue;
        b.emplace_back();
        b.back().R = R[i];
        b.back().F = F[i];
    }
    if (b.empty()) return cudaSuccess;
    const size_t nb = b.size();
    cudaError_t e = cudaSuccess;
    for (size_t i = 0; i < nb && e == cudaSuccess; i++) e = fb_sort(c, b[i]);
    // group counts (and whether a run of a wide key was too long for the
    // run groups) and the error word, one readback
    uint32_t *hg = (uint32_t *)c.pinned;
    std::vector<int64_t> G(nb, 0);
    for (int round = 0; round < 2 && e == cudaSuccess; round++) {
        for (size_t i = 0; i < nb; i++) hg[nb + i] = 0;
        for (size_t i = 0; i < nb && e == cudaSuccess; i++) {
            if (b[i].gcount) e = cudaMemcpyAsync(hg + i, b[i].gcount, sizeof(uint32_t), cudaMemcpyDeviceToHost, c.stream);
            if (e == cudaSuccess && b[i].too_long)
                e = cudaMemcpyAsync(hg + nb + i, b[i].too_long, sizeof(uint32_t), cudaMemcpyDeviceToHost, c.stream);
        }
        if (e == cudaSuccess) e = read_err(hg + 2 * nb);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c.stream);
        if (e != cudaSuccess) break;
        *err_word |= hg[2 * nb];
        bool redo = false;
        for (size_t i = 0; i < nb; i++) {
            G[i] = b[i].gcount ? (int64_t)hg[i] : 0;
            if (hg[nb + i]) {
                // a run longer than the run groups take: build it the two-word way
                Relation *r = b[i].R;
                Factor *f = b[i].F;
                fb_free(c, b[i]);
                factor_free(c, *f);
                b[i] = FactorBuild{};
                b[i].R = r;
                b[i].F = f;
                b[i].force_two = true;
                if (e == cudaSuccess) e = fb_sort(c, b[i]);
                redo = true;
            }
        }
        if (!redo) break;
    }
    for (size_t i = 0; i < nb && e == cudaSuccess; i++) e = fb_groups(c, b[i], G[i]);
    // a factor is handed out complete: a server's slots and queries with a
    // stream of their own read it without waiting on this stream
    if (e == cudaSuccess) e = cudaStreamSynchronize(c.stream);
    if (e != cudaSuccess) {
        note_cuda_error(e, __FILE__, __LINE__);
        for (auto &x : b) fb_free(c, x);
    }
    return e;
}

}  // namespace gj

namespace gj {

cudaError_t radix_sort_u64_u32_in(Ctx &c, uint64_t *keys, uint32_t *vals, int64_t n, int bits,
                                  uint64_t *k2, uint32_t *v2, uint32_t *hist,
                                  unsigned long long *status, int64_t status_tiles);
cudaError_t scan_u32_in(Ctx &c, const uint32_t *in, const uint8_t *flags, uint32_t *out,
                        int64_t n, uint32_t *total_dev, void *state_mem, size_t state_bytes);

// Factor construction of key columns `cols` (device, n rows) with every
// scratch buffer supplied by the caller (no device allocation).  Writes
// perm[n], gstart[G+1] and gkey[nk*G] (column c of group g at c*G + g) and
// *G_out.  Same steps and kernels as factor_build.
cudaError_t factor_build_in(Ctx &c, const int32_t *const *cols, int nk, int64_t n,
                            const std::vector<int> &order, uint32_t *perm, uint32_t *gstart,
                            int32_t *gkey, int64_t *G_out, const FactorScratch &s) {
    *G_out = 0;
    if (n == 0) return cudaMemsetAsync(gstart, 0, sizeof(uint32_t), c.stream);
    ColSet all{};
    all.ncol = nk;
    for (int i = 0; i < nk; i++) all.col[i] = cols[i];
    // 1. min/max per column, read back through host memory on the stack
    k_minmax_init<<<1, 32, 0, c.stream>>>(nk, s.mm); c.launches++;
    const dim3 grid(minmax_blocks(c, n, nk), nk);
    k_minmax<<<grid, FT, 0, c.stream>>>(all, n, s.mm); c.launches++;
    GJ_CUDA_TRY(cudaGetLastError());
    int32_t mm[2 * MAX_KEYS];
    GJ_CUDA_TRY(cudaMemcpyAsync(mm, s.mm, sizeof(int32_t) * 2 * nk, cudaMemcpyDeviceToHost, c.stream));
    GJ_CUDA_TRY(cudaStreamSynchronize(c.stream));
    std::vector<int> bits(nk);
    for (int i = 0; i < nk; i++) bits[i] = bits_of((uint32_t)((int64_t)mm[2 * i + 1] - (int64_t)mm[2 * i]));
    // 2. packed words, least significant first, each sorted stably
    std::vector<std::vector<int>> words;
    {
        std::vector<int> cur;
        int used = 0;
        for (int i = (int)order.size() - 1; i >= 0; i--) {
            int col = order[i];
            if (used + bits[col] > 64 && !cur.empty()) {
                words.push_back(cur);
                cur.clear();
                used = 0;
            }
            cur.push_back(col);
            used += bits[col];
        }
        if (!cur.empty()) words.push_back(cur);
    }
    bool first = true;
    for (auto &wcols : words) {
        PackSpec ps{};
        ps.ncol = (int)wcols.size();
        int shift = 0;
        for (int i = 0; i < ps.ncol; i++) {
            int col = wcols[i];
            ps.col[i] = cols[col];
            ps.mn[i] = mm[2 * col];
            ps.shift[i] = shift;
            shift += bits[col];
        }
        k_pack<<<grid_for(c, n), FT, 0, c.stream>>>(ps, first ? nullptr : perm, n, s.keys, perm); c.launches++;
        GJ_CUDA_TRY(cudaGetLastError());
        GJ_CUDA_TRY(radix_sort_u64_u32_in(c, s.keys, perm, n, shift, s.k2, s.v2, s.hist, s.status,
                                          s.status_tiles));
        first = false;
    }
    // 3. group heads and ids
    if (words.size() == 1) {
        k_heads_packed<<<grid_for(c, n), FT, 0, c.stream>>>(s.keys, n, s.head); c.launches++;
    } else {
        k_heads_gather<<<grid_for(c, n), FT, 0, c.stream>>>(all, perm, n, s.head); c.launches++;
    }
    GJ_CUDA_TRY(cudaGetLastError());
    GJ_CUDA_TRY(scan_u32_in(c, nullptr, s.head, s.gid, n, s.gcount, s.scan_state, s.scan_state_bytes));
    uint32_t G = 0;
    GJ_CUDA_TRY(cudaMemcpyAsync(&G, s.gcount, sizeof(uint32_t), cudaMemcpyDeviceToHost, c.stream));
    GJ_CUDA_TRY(cudaStreamSynchronize(c.stream));
    // 4. group starts and key values
    k_group_compact<<<grid_for(c, n), FT, 0, c.stream>>>(all, perm, s.head, s.gid, n, G, gstart,
                                                         gkey); c.launches++;
    GJ_CUDA_TRY(cudaGetLastError());
    *G_out = G;
    return cudaSuccess;
}

}  // namespace gj

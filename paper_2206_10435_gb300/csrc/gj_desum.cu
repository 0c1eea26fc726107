// gj_desum.cu -- desummarisation (Section 3.6) and summary levels (Def. 1).
//
// The summary places every key path (one group per relation, linked through
// the separators) at a known offset of the sorted result: the root group's
// off, plus, walking the relations in preorder, unit * rel_off of the chosen
// group, where unit is the number of result rows each "way" of that group
// stands for (the p_bucket * bucket product of Algorithm 4 times the ways of
// the subtrees still open beside it).  A window [row0, row0 + n) of the
// result is produced in two steps:
//
//   expand  Algorithm 4 restricted to the window, breadth first: a frontier
//           of path prefixes that overlap the window is extended one
//           relation at a time by the live groups of the linked segment that
//           overlap the window.  Each level is a single-pass scan that counts
//           every prefix's groups and numbers their slots, and a load-balanced
//           write kernel (a CTA owns a tile of output slots and maps them to
//           prefixes by a shared-memory search), so a segment with 10^5
//           groups costs no more than 10^5 tiny ones.
//   emit    every result row finds its block (full key path) by a binary
//           search of the block offsets staged in shared memory, splits its
//           offset inside the block into one row index per relation (mixed
//           radix, relation 1 most significant: rows of a block are ordered
//           by r_1..r_k) and writes the key values (block constants) and the
//           payloads, gathered from the factors' group-ordered copies.
//           Consecutive threads write consecutive rows of each column.
//
// A level of the paper's GFJS (Figure 2) is the run list of the frontier at
// the relation that introduces the level's variable.
#include <algorithm>

#include "gj_emit.cuh"
#include "gj_lookback.cuh"

namespace gj {

gj_status check_device_error(Ctx &c);

namespace {

constexpr int DT = 256;          // threads per CTA
constexpr int EXP_TILE = 1024;   // output slots per CTA in expansion
constexpr int EMIT_TILE = 1024;  // result rows per CTA in emission

// One frontier: path prefixes (groups of preorder relations 0..depth-1).
// Arrays are sized for `cap` items; the item count lives in device memory.
// They are parts of the expansion's one block, held by the frontier handed out.
struct Frontier {
    int64_t cap = 0;
    Workspace::Block own{};
    uint32_t *F_dev = nullptr;           // number of items
    uint64_t *A = nullptr;               // absolute first result row
    uint64_t *W = nullptr;               // product of the chosen groups' counts
    uint32_t *grp[MAX_REL] = {};         // grp[p][i]: group of preorder relation p
    uint32_t *lh = nullptr;              // live index of the last group (optional)
    uint64_t *unit = nullptr;            // rows per way of the last group (optional)
    void *spare = nullptr;               // the caller may use: 4 B per item, and cleared
    unsigned long long *state = nullptr; // lookback state for one scan of the items, from word 1 on
};

void frontier_free(Ctx &c, Frontier &f) {
    ws_give(c, WS_TEMP, f.own);
}

constexpr int MAXR = MAX_REL;

// Everything an expansion step needs, by value.
struct ExpandSpec {
    // relation being added (preorder index j)
    const uint32_t *link;          // parent's link to it, indexed by parent group
    int parent_p;                  // preorder index of its parent
    const uint32_t *lseg_first;    // [S+1]
    const uint64_t *msg;           // [S]
    const uint32_t *lgid;
    const uint64_t *loff;          // rel_off of live groups
    const uint64_t *lw;
    const uint32_t *gstart;
    // open subtrees beside it: multiply unit by their message
    int nrest;
    const uint32_t *rest_link[MAXR];
    const uint64_t *rest_msg[MAXR];
    int rest_parent_p[MAXR];
    // frontier in
    int depth;                     // = j
    const uint64_t *A, *W;
    const uint32_t *grp[MAXR];
    uint32_t *err;
};

__device__ __forceinline__ uint64_t item_unit(const ExpandSpec &s, int64_t i) {
    uint64_t u = s.W[i];
    for (int r = 0; r < s.nrest; r++) {
        uint32_t g = s.grp[s.rest_parent_p[r]][i];
        uint32_t seg = s.rest_link[r][g];
        u = sat_mul(u, seg == NONE ? 0ull : s.rest_msg[r][seg]);
    }
    return u;
}

// first h in [a, b) with key(h) > x, key non-decreasing
template <class F>
__device__ __forceinline__ uint32_t first_greater(uint32_t a, uint32_t b, uint64_t x, F key) {
    while (a < b) {
        uint32_t m = a + ((b - a) >> 1);
        if (key(m) > x) b = m; else a = m + 1;
    }
    return a;
}

// first index h in [a, b) with key(h) > x (key non-decreasing), by one warp:
// each round the 32 lanes probe 32 evenly spaced points and the interval
// shrinks to the gap between two of them (about log32 of the length rounds)
template <class F>
__device__ __forceinline__ uint32_t warp_first_greater(uint32_t a, uint32_t b, uint64_t x, F key) {
    const int lane = threadIdx.x & 31;
    while (b - a > 32) {
        const uint32_t step = (b - a + 31) / 32;
        const uint32_t p = a + lane * step;   // lane 0 probes a
        const bool gt = p < b && key(p) > x;
        const uint32_t m = __ballot_sync(0xffffffffu, gt);
        // the answer lies in (probe of the last lane not greater, probe of the first greater]
        const int f = m ? __ffs((int)m) - 1 : 32;   // first probing lane with key > x
        if (f == 0) return a;                        // key(a) > x
        if (f == 32) {                               // none greater: past the last probe inside
            a += ((b - 1 - a) / step) * step + 1;
        } else {                                     // between probes f - 1 and f
            b = a + (uint32_t)f * step;
            a += (uint32_t)(f - 1) * step + 1;
        }
    }
    const uint32_t p = a + lane;
    const bool gt = p < b && key(p) > x;
    const uint32_t m = __ballot_sync(0xffffffffu, gt);
    return m ? a + (uint32_t)(__ffs((int)m) - 1) : b;
}

// The root of an expansion: its live groups in result order.
struct RootSpec {
    const uint32_t *lgid;
    const uint64_t *loff, *lw;
    const uint32_t *gstart;
    const uint32_t *L_dev;
    // the frontier over the root alone, written for the window's groups
    uint64_t *A, *W;
    uint32_t *grp0;
    uint32_t *lh;                  // optional, with unit
    uint64_t *unit;
    uint32_t *F_dev;
};

// The live root groups h whose rows [loff, loff + lw) overlap the window:
// found by one warp of the calling CTA (two searches, a few rounds of probes).
__device__ __forceinline__ void root_range(const RootSpec &r, uint64_t row0, uint64_t row_end, uint32_t *lo,
                                           uint32_t *hi) {
    const uint32_t L = *r.L_dev;
    const uint32_t a = warp_first_greater(0u, L, row0, [&](uint32_t h) { return r.loff[h] + r.lw[h]; });
    const uint32_t b = warp_first_greater(a, L, row_end - 1, [&](uint32_t h) { return r.loff[h]; });
    if ((threadIdx.x & 31) == 0) {
        *lo = a;
        *hi = b;
    }
}

// the frontier of an expansion that stops at the root
__global__ void __launch_bounds__(DT) k_root_frontier(RootSpec r, uint64_t row0, uint64_t row_end) {
    __shared__ uint32_t s_lo, s_hi;
    if (threadIdx.x < 32) root_range(r, row0, row_end, &s_lo, &s_hi);
    __syncthreads();
    const uint32_t lo = s_lo;
    const int64_t F = s_hi - lo;
    if (blockIdx.x == 0 && threadIdx.x == 0) *r.F_dev = (uint32_t)F;
    for (int64_t i = (int64_t)blockIdx.x * DT + threadIdx.x; i < F; i += (int64_t)gridDim.x * DT) {
        const uint32_t h = lo + (uint32_t)i;
        const uint32_t g = r.lgid[h];
        r.A[i] = r.loff[h];
        if (r.W) r.W[i] = (uint64_t)(r.gstart[g + 1] - r.gstart[g]);
        r.grp0[i] = g;
        if (r.lh) r.lh[i] = h;
        if (r.unit) r.unit[i] = 1;
    }
}

// Where an item's slots go, for the write kernel.
struct ExpandScanOut {
    uint32_t *excl, *lo;           // first slot; live index of the first group
    uint64_t *unit;
    uint32_t *slot_first;          // [t]: item owning slot t * EXP_TILE
    uint32_t *Fout;                // slots in all
    uint32_t *counter;             // lookback state, cleared beforehand
    unsigned long long *status;
};

constexpr int EC_ITEMS = 4;
constexpr int EC_TILE = DT * EC_ITEMS;

// One level's counts and slots in a single pass: per item the live groups of
// its linked segment that overlap the window (count, first live index, rows per
// way), their exclusive prefix (decoupled lookback over tiles taken in order by
// a resident grid; the item count is in device memory), and the slot tiles'
// owners.  With ROOT the items are the root's live groups of the window, found
// and written out here too.  Bound by the dependent gathers behind each item's
// group (link, segment bounds, message), four items per thread in flight.  A
// level was a count, a scan, a slot map and a cleared state (for the first, a
// range search and an init kernel too): six run-length columns of a window of
// 2e7 rows 1.11 -> 0.51 ms with 98 -> 46 device operations and 182 -> 0
// allocations; 5-chain window of 1e8 rows 119 -> 115 us in these kernels.
template <bool ROOT>
__global__ void __launch_bounds__(DT)
k_expand_scan(ExpandSpec s, RootSpec r, const uint32_t *F_dev, uint64_t row0, uint64_t row_end, ExpandScanOut o) {
    __shared__ uint32_t s_lo, s_hi, s_tile, s_carry;
    __shared__ uint32_t s_warp[DT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t root_lo = 0;
    int64_t F;
    if (ROOT) {
        if (warp == 0) root_range(r, row0, row_end, &s_lo, &s_hi);
        __syncthreads();
        root_lo = s_lo;
        F = s_hi - root_lo;
    } else {
        F = *F_dev;
    }
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(o.counter, 1u);
        __syncthreads();
        const uint32_t tile = s_tile;
        const int64_t base = (int64_t)tile * EC_TILE;
        if (tile == 0 && tid == 0) {
            if (ROOT) *r.F_dev = (uint32_t)F;
            if (F == 0) *o.Fout = 0;
        }
        if (base >= F) return;
        // items of a warp are consecutive: item (i, lane) at i * 32 + lane
        const int64_t wbase = base + warp * (32 * EC_ITEMS) + lane;
        uint32_t gp[EC_ITEMS], seg[EC_ITEMS], a[EC_ITEMS], b[EC_ITEMS], cnt[EC_ITEMS], lo[EC_ITEMS];
        uint64_t A[EC_ITEMS], unit[EC_ITEMS];
#pragma unroll
        for (int i = 0; i < EC_ITEMS; i++) {
            const int64_t t = wbase + i * 32;
            gp[i] = 0;
            A[i] = 0;
            if (t < F) {
                if (ROOT) {
                    gp[i] = r.lgid[root_lo + (uint32_t)t];
                    A[i] = r.loff[root_lo + (uint32_t)t];
                } else {
                    gp[i] = s.grp[s.parent_p][t];
                    A[i] = s.A[t];
                }
            }
        }
#pragma unroll
        for (int i = 0; i < EC_ITEMS; i++) {
            const int64_t t = wbase + i * 32;
            seg[i] = NONE;
            unit[i] = 1;
            if (t < F) {
                seg[i] = s.link[gp[i]];
                if (ROOT) {
                    // one root group per item: its count, and its other subtrees
                    uint64_t u = (uint64_t)(r.gstart[gp[i] + 1] - r.gstart[gp[i]]);
                    r.A[t] = A[i];
                    r.W[t] = u;
                    r.grp0[t] = gp[i];
                    for (int k = 0; k < s.nrest; k++) {
                        const uint32_t sg = s.rest_link[k][gp[i]];
                        u = sat_mul(u, sg == NONE ? 0ull : s.rest_msg[k][sg]);
                    }
                    unit[i] = u;
                } else {
                    unit[i] = item_unit(s, t);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < EC_ITEMS; i++) {
            a[i] = b[i] = 0;
            if (seg[i] != NONE) {
                a[i] = s.lseg_first[seg[i]];
                b[i] = s.lseg_first[seg[i] + 1];
            }
        }
#pragma unroll
        for (int i = 0; i < EC_ITEMS; i++) {
            const int64_t t = wbase + i * 32;
            cnt[i] = lo[i] = 0;
            if (t >= F) continue;
            if (seg[i] == NONE) { raise_err(s.err, ERRF_BOUNDS); unit[i] = 1; continue; }
            uint32_t first = a[i], last = b[i];
            if (A[i] < row0) {
                const uint64_t X = (row0 - A[i]) / unit[i];   // need unit * (off + w) > row0 - A
                first = first_greater(a[i], b[i], X, [&](uint32_t h) { return s.loff[h] + s.lw[h]; });
            }
            const uint64_t end = A[i] + unit[i] * s.msg[seg[i]];
            if (end > row_end) {
                const uint64_t Y = (row_end - 1 - A[i]) / unit[i];   // need unit * off <= row_end - 1 - A
                last = first_greater(a[i], b[i], Y, [&](uint32_t h) { return s.loff[h]; });
            }
            if (last < first) { raise_err(s.err, ERRF_BOUNDS); last = first; }
            cnt[i] = last - first;
            lo[i] = first;
        }
        // exclusive prefix of the counts, in item order
        uint32_t ex[EC_ITEMS], run = 0;
#pragma unroll
        for (int i = 0; i < EC_ITEMS; i++) {
            uint32_t x = cnt[i];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
                if (lane >= d) x += y;
            }
            ex[i] = run + x - cnt[i];
            run += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) s_warp[warp] = run;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < warp; w++) before += s_warp[w];
        if (warp == DT / 32 - 1) {
            const uint32_t agg = before + run;
            const uint32_t carry = warp_lookback<uint32_t, AddU32>(o.status, tile, agg, lane, s.err);
            if (lane == 0) {
                s_carry = carry;
                if (base + EC_TILE >= F) *o.Fout = carry + agg;
            }
        }
        __syncthreads();
        const uint32_t carry = s_carry + before;
#pragma unroll
        for (int i = 0; i < EC_ITEMS; i++) {
            const int64_t t = wbase + i * 32;
            if (t >= F) continue;
            const uint32_t e = carry + ex[i];
            o.excl[t] = e;
            o.lo[t] = lo[i];
            o.unit[t] = unit[i];
            const uint64_t end = (uint64_t)e + cnt[i];
            for (uint64_t x = ((uint64_t)e + EXP_TILE - 1) / EXP_TILE; x * EXP_TILE < end; x++)
                o.slot_first[x] = (uint32_t)t;
        }
        __syncthreads();   // s_warp and s_carry are free for the next tile
    }
}

struct ExpandOut {
    uint64_t *A, *W;
    uint32_t *grp[MAXR];
    uint32_t *lh;
    uint64_t *unit;
    // last level of a desummarisation: tile_first[t] = block holding window
    // row t * tile_rows (the emit's tile map), written by the blocks
    uint32_t *tile_first;
    int64_t tile_rows, tiles;
    uint64_t row0;
    int64_t n;
};

// Tiles of EXP_TILE output slots, taken in turn by a persistent grid (the
// number of tiles follows from the next frontier's size in device memory);
// slot -> source item by a search of the item offsets staged in shared
// memory (each item has >= 1 slot).
__global__ void __launch_bounds__(DT)
k_expand_write(ExpandSpec s, const uint32_t *F_dev, const uint32_t *__restrict__ excl,
               const uint32_t *Fout_dev, const uint32_t *__restrict__ slot_first,
               const uint32_t *__restrict__ lo_in, const uint64_t *__restrict__ unit_in,
               ExpandOut o) {
    __shared__ uint32_t s_off[EXP_TILE + 1];
    __shared__ uint64_t s_A[EXP_TILE];   // tile map only: first rows of the tile's blocks
    __shared__ uint64_t s_end;            // and the end of its last block
    const int64_t F = *F_dev, Fout = *Fout_dev;
    const int64_t tiles = (Fout + EXP_TILE - 1) / EXP_TILE;
    const int j = s.depth;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t o0 = tile * EXP_TILE;
        const int64_t o1 = min(Fout, o0 + EXP_TILE);
        const int64_t first = slot_first[tile];
        const int64_t last = (tile + 1 < tiles) ? (int64_t)slot_first[tile + 1] : F - 1;
        const int nitems = (int)(last - first + 1);
        // every item owns >= 1 slot, so a tile sees at most EXP_TILE + 1 items
        if (last < first || nitems > EXP_TILE + 1) {
            if (threadIdx.x == 0) raise_err(s.err, ERRF_BOUNDS);
            return;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < nitems; t += DT) s_off[t] = excl[first + t];
        __syncthreads();
        for (int64_t slot = o0 + threadIdx.x; slot < o1; slot += DT) {
            int a = 0, b = nitems;   // last t with s_off[t] <= slot
            while (a < b) { int m = (a + b) >> 1; if (s_off[m] <= (uint32_t)slot) a = m + 1; else b = m; }
            const int64_t i = first + a - 1;
            const uint32_t h = lo_in[i] + (uint32_t)(slot - s_off[a - 1]);
            const uint32_t g = s.lgid[h];
            const uint64_t unit = unit_in[i];
            const uint64_t A = s.A[i] + unit * s.loff[h];
            o.A[slot] = A;
            if (o.W) o.W[slot] = s.W[i] * (uint64_t)(s.gstart[g + 1] - s.gstart[g]);
            if (o.tile_first) {
                s_A[slot - o0] = A;
                // the tile's last block ends where the next tile starts: its
                // size is needed
                if (slot == o1 - 1) s_end = A + s.W[i] * (uint64_t)(s.gstart[g + 1] - s.gstart[g]);
            }
            for (int p = 0; p < j; p++) o.grp[p][slot] = s.grp[p][i];
            o.grp[j][slot] = g;
            if (o.lh) o.lh[slot] = h;
            if (o.unit) o.unit[slot] = unit;
        }
        if (o.tile_first) {
            // the tile's blocks hold rows [s_A[0], s_end) of the result: every
            // emit tile whose first row lies there points at the block holding
            // that row (threads take tiles, not blocks, so one huge block
            // costs no single thread more than its share)
            __syncthreads();
            const int64_t T = o.tile_rows;
            const int ns = (int)(o1 - o0);
            const uint64_t lo = s_A[0] > o.row0 ? s_A[0] - o.row0 : 0;
            const uint64_t hi = min(s_end - o.row0, (uint64_t)o.n);
            const int64_t t0 = (int64_t)((lo + T - 1) / T), t1 = min(o.tiles, (int64_t)((hi + T - 1) / T));
            // blocks with first row <= that of emit tile t, of which the first
            // `a` are known to be
            auto upto = [&](int64_t t, int a) {
                const uint64_t row = o.row0 + (uint64_t)(t * T);
                int b = ns;
                while (a < b) { int m = (a + b) >> 1; if (s_A[m] <= row) a = m + 1; else b = m; }
                return a;
            };
            if (t1 - t0 <= 4 * DT) {
                for (int64_t t = t0 + threadIdx.x; t < t1; t += DT) o.tile_first[t] = (uint32_t)(o0 + upto(t, 0) - 1);
            } else {
                // large blocks: four emit tiles per thread and round, which
                // mostly point at the block of the round before
                int a = 0;
                for (int64_t b = t0 / 4 * 4 + 4 * threadIdx.x; b < t1; b += 4 * DT) {
                    uint32_t v[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        if (a < ns && s_A[a] <= o.row0 + (uint64_t)((b + u) * T)) a = upto(b + u, a);
                        v[u] = (uint32_t)(o0 + a - 1);
                    }
                    if (b >= t0 && b + 4 <= t1) {
                        *(uint4 *)(o.tile_first + b) = make_uint4(v[0], v[1], v[2], v[3]);
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; u++)
                            if (b + u >= t0 && b + u < t1) o.tile_first[b + u] = v[u];
                    }
                }
            }
        }
    }
}

inline int grid_for(Ctx &c, int64_t n) {
    int64_t b = ceil_div(n, DT);
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, (int64_t)c.num_sms * 16));
}

cudaError_t readback(Ctx &c, const void *dev, void *host, size_t bytes) {
    GJ_CUDA_TRY(cudaMemcpyAsync(c.pinned, dev, bytes, cudaMemcpyDeviceToHost, c.stream));
    GJ_CUDA_TRY(cudaStreamSynchronize(c.stream));
    memcpy(host, c.pinned, bytes);
    return cudaSuccess;
}

// The open subtrees beside preorder step j (see item_unit): simulate the DFS
// stack of the preorder walk.
std::vector<int> rest_at(const QueryState &q, int j) {
    std::vector<int> open(q.r[q.pre[0]].children);
    for (int step = 1; step <= j; step++) {
        int t = q.pre[step];
        // preorder: t is the top of the stack
        std::vector<int> next(q.r[t].children);
        next.insert(next.end(), open.begin() + 1, open.end());
        if (step == j) return std::vector<int>(open.begin() + 1, open.end());
        open.swap(next);
    }
    return {};
}

int child_index(const QRel &parent, int child_pos) {
    for (size_t i = 0; i < parent.children.size(); i++)
        if (parent.children[i] == child_pos) return (int)i;
    return -1;
}

// Frontier of path prefixes through preorder relations 0..depth-1 that
// overlap result rows [row0, row_end).  No host synchronisation: every
// frontier holds at most one item per row of the window, so arrays are
// sized by the window and item counts stay in device memory.
// keep_last: also fill lh and unit.  tm: the last level also writes the emit
// kernel's tile map (the block holding the first row of every emit tile).
struct TileMap {
    uint32_t *tile_first;   // [tiles + 1]
    int64_t tile_rows, tiles;
};

// All arrays of an expansion are parts of one block: every level's lookback
// state, two frontiers that the levels alternate between, and the scans' outputs.
// (A level had seven arrays of its own; for small windows their allocation calls
// took longer than the kernels.)  A level's frontier is dead once the next one
// is written, so a level writes over the one before the last; the last level has
// no W, and its last two group columns take that array's place.  So a window of
// chains of 2, 3, 4 and 5 relations takes 52, 60, 68 and 76 bytes a row.
cudaError_t expand(QueryState &q, uint64_t row0, uint64_t row_end, int depth, bool keep_last,
                   Frontier &out, const TileMap *tm = nullptr) {
    Ctx &c = q.ctx();
    const QRel &root = q.r[q.pre[0]];
    const int64_t cap = (int64_t)(row_end - row0);
    const int64_t cap0 = std::min(cap, std::max<int64_t>(root.F->G, 1));   // the root's frontier
    const int64_t slot_tiles = ceil_div(cap, EXP_TILE), scan_tiles = ceil_div(cap, EC_TILE);
    auto resident = [&](int64_t tiles) { return (int)std::max<int64_t>(1, std::min<int64_t>(tiles, c.num_sms * 8)); };
    struct Hold {
        Ctx &c;
        Frontier f;
        ~Hold() { frontier_free(c, f); }
    } hold{c, {}};
    std::vector<std::pair<void **, size_t>> want;
    // 64-bit words of a 32-bit array of n entries, aligned like the parts
    auto w_half = [](int64_t n) { return (n * 4 + 255) / 256 * 32; };
    auto add = [&](auto **p, size_t count) { want.emplace_back((void **)p, (count * sizeof(**p) + 255) & ~(size_t)255); };
    // per frontier: its count, and the tile counter and status words of the scan
    // over it (the caller's, for the last one); all cleared at once
    const size_t state_words = 2 + (size_t)scan_tiles;
    unsigned long long *state = nullptr;
    const int last = depth - 1;
    Frontier lev[2];                     // level l is in lev[l & 1]
    ExpandScanOut so{};
    uint32_t *spare = nullptr;
    add(&state, state_words * (size_t)depth);
    for (int p = 0; p < 2 && p <= last; p++) {
        Frontier &f = lev[p];
        const bool ends = (last & 1) == p;
        const int top = ends ? last - 2 : last - 1;   // its last level but the last of all
        f.cap = ends ? (last > 0 ? cap : cap0) : (top > 0 ? cap : cap0);
        add(&f.A, f.cap);
        const int own = top >= 0 ? top : last;
        for (int g = 0; g <= own; g++) add(&f.grp[g], f.cap);
        if (top >= 0) add(&f.W, ends ? 2 * w_half(f.cap) : f.cap);
        if (ends && keep_last) {
            add(&f.lh, f.cap);
            add(&f.unit, f.cap);
            add(&spare, f.cap);
        }
    }
    if (depth > 1) {
        const int64_t items = depth > 2 ? cap : cap0;
        add(&so.lo, items);
        add(&so.excl, items);
        add(&so.unit, items);
        add(&so.slot_first, slot_tiles + 1);
    }
    size_t bytes = 0;
    for (auto &w : want) bytes += w.second;
    GJ_CUDA_TRY(ws_take(c, WS_TEMP, bytes, &hold.f.own));
    char *at = (char *)hold.f.own.p;
    for (auto &w : want) {
        *w.first = at;
        at += w.second;
    }
    if (last >= 2) {
        Frontier &f = lev[last & 1];
        f.grp[last - 1] = (uint32_t *)f.W;
        f.grp[last] = (uint32_t *)(f.W + w_half(f.cap));
    }
    // a level's frontier: its capacity, count and the arrays it has
    auto level = [&](int l) {
        Frontier f = lev[l & 1];
        f.cap = l == 0 ? cap0 : cap;
        f.F_dev = (uint32_t *)(state + state_words * (size_t)l);
        if (l == last) f.W = nullptr;
        else f.lh = nullptr, f.unit = nullptr;
        return f;
    };
    GJ_CUDA_TRY(cudaMemsetAsync(state, 0, 8 * state_words * (size_t)depth, c.stream));
    auto state_of = [&](int level) { return state + state_words * (size_t)level; };
    Frontier cur = level(0);
    RootSpec rs{};
    rs.lgid = root.lgid;
    rs.loff = root.loff;
    rs.lw = root.lw;
    rs.gstart = root.F->gstart;
    rs.L_dev = root.L_dev;
    rs.A = cur.A;
    rs.W = cur.W;
    rs.grp0 = cur.grp[0];
    rs.lh = cur.lh;
    rs.unit = cur.unit;
    rs.F_dev = cur.F_dev;
    if (depth == 1) {
        k_root_frontier<<<grid_for(c, cap), DT, 0, c.stream>>>(rs, row0, row_end); c.launches++;
        GJ_CUDA_TRY(cudaGetLastError());
    }
    for (int j = 1; j < depth; j++) {
        const int tpos = q.pre[j];
        const QRel &t = q.r[tpos];
        const QRel &par = q.r[t.parent];
        ExpandSpec s{};
        s.link = par.link[child_index(par, tpos)];
        s.parent_p = q.pos[t.parent];
        s.lseg_first = t.lseg_first;
        s.msg = t.msg;
        s.lgid = t.lgid;
        s.loff = t.loff;
        s.lw = t.lw;
        s.gstart = t.F->gstart;
        std::vector<int> rest = rest_at(q, j);
        s.nrest = (int)rest.size();
        for (int r = 0; r < s.nrest; r++) {
            const QRel &rc = q.r[rest[r]];
            const QRel &rp = q.r[rc.parent];
            s.rest_link[r] = rp.link[child_index(rp, rest[r])];
            s.rest_msg[r] = rc.msg;
            s.rest_parent_p[r] = q.pos[rc.parent];
        }
        s.depth = j;
        s.err = c.err;
        s.A = cur.A;
        s.W = cur.W;
        for (int p = 0; p < j; p++) s.grp[p] = cur.grp[p];
        ExpandScanOut e = so;
        e.Fout = (uint32_t *)state_of(j);
        e.counter = (uint32_t *)(state_of(j - 1) + 1);
        e.status = state_of(j - 1) + 2;
        const int sgrid = resident(ceil_div(cur.cap, EC_TILE));
        if (j == 1) k_expand_scan<true><<<sgrid, DT, 0, c.stream>>>(s, rs, nullptr, row0, row_end, e);
        else k_expand_scan<false><<<sgrid, DT, 0, c.stream>>>(s, rs, cur.F_dev, row0, row_end, e);
        c.launches++;
        GJ_CUDA_TRY(cudaGetLastError());
        Frontier nxt = level(j);
        ExpandOut o{};
        o.A = nxt.A;
        o.W = nxt.W;
        for (int p = 0; p <= j; p++) o.grp[p] = nxt.grp[p];
        o.lh = nxt.lh;
        o.unit = nxt.unit;
        if (j == last && tm) {
            o.tile_first = tm->tile_first;
            o.tile_rows = tm->tile_rows;
            o.tiles = tm->tiles;
            o.row0 = row0;
            o.n = (int64_t)(row_end - row0);
        }
        k_expand_write<<<resident(slot_tiles), DT, 0, c.stream>>>(s, cur.F_dev, e.excl, nxt.F_dev, e.slot_first,
                                                                  e.lo, e.unit, o); c.launches++;
        GJ_CUDA_TRY(cudaGetLastError());
        cur = nxt;
    }
    std::swap(cur.own, hold.f.own);
    cur.spare = spare;
    cur.state = state_of(depth - 1);
    out = std::move(cur);
    return cudaSuccess;
}

// ------------------------------------------------------------------ emission

constexpr int MAXV = 32;
constexpr int MAXP = 32;

struct EmitSpec {
    int k;                                // relations (query positions)
    int preidx[MAXR];                     // query position -> preorder index
    const uint32_t *gstart[MAXR];
    const uint32_t *perm[MAXR];
    uint32_t *rid_out[MAXR];
    int nv;
    const int32_t *vkey[MAXV];            // gkey row of the V column
    int vrel[MAXV];                       // query position owning it
    int32_t *vout[MAXV];
    int np;
    const void *pay[MAXP];
    int prel[MAXP];
    int pw[MAXP];
    void *pout[MAXP];
    const uint64_t *A;                    // block offsets
    const uint32_t *grp[MAXR];            // by preorder index
    uint32_t *err;
};

__global__ void __launch_bounds__(DT)
k_emit(EmitSpec e, const uint32_t *B_dev, uint64_t row0, int64_t n) {
    const int64_t B = *B_dev;
    __shared__ uint64_t s_A[EMIT_TILE + 1];
    __shared__ int64_t s_first;
    __shared__ int s_cnt;
    const int64_t r0 = (int64_t)blockIdx.x * EMIT_TILE;
    if (r0 >= n) return;
    const int64_t r1 = min(n, r0 + EMIT_TILE);
    if (threadIdx.x == 0) {
        int64_t a = 0, b = B;
        uint64_t x = row0 + (uint64_t)r0;
        while (a < b) { int64_t m = (a + b) >> 1; if (e.A[m] <= x) a = m + 1; else b = m; }
        int64_t first = a - 1;
        x = row0 + (uint64_t)(r1 - 1);
        a = first; b = B;
        while (a < b) { int64_t m = (a + b) >> 1; if (e.A[m] <= x) a = m + 1; else b = m; }
        s_first = first;
        int64_t cnt = a - first;
        if (first < 0 || cnt > EMIT_TILE) { raise_err(e.err, ERRF_BOUNDS); cnt = 0; }
        s_cnt = (int)cnt;
    }
    __syncthreads();
    const int64_t first = s_first;
    const int nb = s_cnt;
    if (nb == 0) return;
    for (int t = threadIdx.x; t < nb; t += DT) s_A[t] = e.A[first + t];
    __syncthreads();
    for (int64_t r = r0 + threadIdx.x; r < r1; r += DT) {
        const uint64_t row = row0 + (uint64_t)r;
        int a = 0, b = nb;
        while (a < b) { int m = (a + b) >> 1; if (s_A[m] <= row) a = m + 1; else b = m; }
        const int64_t blk = first + a - 1;
        uint64_t q = row - s_A[a - 1];
        uint32_t pos[MAXR];
        // mixed radix, relation k-1 fastest
        for (int j = e.k - 1; j >= 0; j--) {
            uint32_t g = e.grp[e.preidx[j]][blk];
            uint32_t base = e.gstart[j][g];
            uint32_t cnt = e.gstart[j][g + 1] - base;
            uint32_t d;
            if (q < 0x100000000ull) { uint32_t q32 = (uint32_t)q; d = q32 % cnt; q = q32 / cnt; }
            else { d = (uint32_t)(q % cnt); q /= cnt; }
            pos[j] = base + d;
        }
        for (int v = 0; v < e.nv; v++) {
            uint32_t g = e.grp[e.preidx[e.vrel[v]]][blk];
            e.vout[v][r] = e.vkey[v][g];
        }
        for (int p = 0; p < e.np; p++) {
            uint32_t at = pos[e.prel[p]];
            if (e.pw[p] == 8) ((uint64_t *)e.pout[p])[r] = ((const uint64_t *)e.pay[p])[at];
            else ((uint32_t *)e.pout[p])[r] = ((const uint32_t *)e.pay[p])[at];
        }
        for (int j = 0; j < e.k; j++)
            if (e.rid_out[j]) e.rid_out[j][r] = e.perm[j][pos[j]];
    }
}

// ------------------------------------------------------------------ levels

struct LevelSpec {
    const uint64_t *A;
    const uint32_t *lh;
    const uint64_t *unit;
    const uint32_t *lgid;
    const uint64_t *loff, *lw;
    const uint32_t *seg_id;       // NULL for the root
    const uint32_t *lseg_first;
    const uint32_t *L_dev;
    int nprefix;                  // new columns up to and including the level's
    bool last;                    // level's column is the relation's last new column
    const int32_t *pcol[MAX_KEYS];
    const int32_t *vcol;
};

__device__ __forceinline__ bool same_prefix(const LevelSpec &s, uint32_t g1, uint32_t g2) {
    for (int c = 0; c < s.nprefix; c++)
        if (s.pcol[c][g1] != s.pcol[c][g2]) return false;
    return true;
}

// The runs among the frontier's items, numbered in one pass: idx[i] = the run
// item i starts, or NONE.  An item of an earlier run of the level, or one that
// starts before the window, starts none.  *runs receives their number.
__global__ void __launch_bounds__(DT)
k_level_scan(LevelSpec s, const uint32_t *F_dev, uint64_t row0, uint32_t *counter, unsigned long long *status,
             uint32_t *idx, uint32_t *runs, uint32_t *err) {
    __shared__ uint32_t s_tile, s_carry, s_warp[DT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t F = *F_dev;
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(counter, 1u);
        __syncthreads();
        const uint32_t tile = s_tile;
        const int64_t base = (int64_t)tile * EC_TILE;
        if (F == 0 && tile == 0 && tid == 0) *runs = 0;
        if (base >= F) return;
        const int64_t wbase = base + warp * (32 * EC_ITEMS) + lane;
        uint32_t h[EC_ITEMS], hb[EC_ITEMS], run = 0;
        uint64_t A[EC_ITEMS];
#pragma unroll
        for (int i = 0; i < EC_ITEMS; i++) {
            const int64_t t = wbase + i * 32;
            A[i] = t < F ? s.A[t] : 0ull;
            h[i] = t < F && !s.last ? s.lh[t] : 0u;   // the last column: every item is a run
        }
#pragma unroll
        for (int i = 0; i < EC_ITEMS; i++) {
            bool f = wbase + i * 32 < F && A[i] >= row0;
            if (f && !s.last) {
                const uint32_t g = s.lgid[h[i]];
                const uint32_t a = s.seg_id ? s.lseg_first[s.seg_id[g]] : 0u;
                f = h[i] == a || !same_prefix(s, s.lgid[h[i] - 1], g);
            }
            hb[i] = __ballot_sync(0xffffffffu, f);
            run += __popc(hb[i]);
        }
        if (lane == 0) s_warp[warp] = run;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < warp; w++) before += s_warp[w];
        if (warp == DT / 32 - 1) {
            const uint32_t agg = before + run;
            const uint32_t carry = warp_lookback<uint32_t, AddU32>(status, tile, agg, lane, err);
            if (lane == 0) {
                s_carry = carry;
                if (base + EC_TILE >= F) *runs = carry + agg;
            }
        }
        __syncthreads();
        uint32_t at = s_carry + before;
        const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
        for (int i = 0; i < EC_ITEMS; i++) {
            const int64_t t = wbase + i * 32;
            if (t < F) idx[t] = (hb[i] >> lane) & 1u ? at + __popc(hb[i] & lt) : NONE;
            at += __popc(hb[i]);
        }
        __syncthreads();
    }
}

// writes nothing when the runs exceed the caller's capacity
__global__ void k_level_write(LevelSpec s, const uint32_t *F_dev, const uint32_t *idx, const uint32_t *runs,
                              uint64_t cap, int32_t *val, uint64_t *freq, uint64_t *off) {
    const int64_t F = *runs <= cap ? *F_dev : 0;
    for (int64_t i = (int64_t)blockIdx.x * DT + threadIdx.x; i < F; i += (int64_t)gridDim.x * DT) {
        const uint32_t o = idx[i];
        if (o == NONE) continue;
        uint32_t h = s.lh[i];
        uint32_t g = s.lgid[h];
        uint32_t he = h;
        if (!s.last) {
            uint32_t b = s.seg_id ? s.lseg_first[s.seg_id[g] + 1] : *s.L_dev;
            uint32_t a = h + 1;   // first live index after h with a different prefix
            while (a < b) {
                uint32_t m = a + ((b - a) >> 1);
                if (same_prefix(s, s.lgid[m], g)) a = m + 1; else b = m;
            }
            he = a - 1;
        }
        val[o] = s.vcol[g];
        freq[o] = s.unit[i] * (s.loff[he] + s.lw[he] - s.loff[h]);
        off[o] = s.A[i];
    }
}

}  // namespace

// The emit kernel's description of a query's output: for every relation
// (query position j) its factor, its block groups grp[j] and its output
// columns (key columns of V, then payloads).  False if the layout exceeds
// the kernel's limits.
bool make_emit_spec(QueryState &q, void *const *out_cols, uint32_t *const *rowid_cols,
                    const uint32_t *const *grp, const uint64_t *A, Emit4Spec &s) {
    s = Emit4Spec{};
    if (q.k > EMIT_MAXR || (int)q.var_rel.size() > EMIT_MAXV || (int)q.col_rel.size() > EMIT_MAXP)
        return false;
    int nc = 0;
    bool vec = true;
    const int nv = (int)q.var_rel.size();
    for (int j = 0; j < q.k; j++) {
        s.gstart[j] = q.r[j].F->gstart;
        s.perm[j] = q.r[j].F->perm;
        s.rid_out[j] = rowid_cols ? rowid_cols[j] : nullptr;
        s.grp[j] = grp[j];
        s.col_off[j] = nc;
        for (int v = 0; v < nv; v++) {
            if (q.var_rel[v] != j) continue;
            s.src[nc] = q.r[j].F->key(q.var_col[v]);
            s.dst[nc] = out_cols[v];
            s.kind[nc] = 0;
            nc++;
        }
        for (size_t p = 0; p < q.col_rel.size(); p++) {
            if (q.col_rel[p] != j) continue;
            s.src[nc] = q.r[j].F->pay[q.col_pay[p]];
            s.dst[nc] = out_cols[nv + p];
            s.kind[nc] = q.r[j].R->pw[q.col_pay[p]] == 8 ? 2 : 1;
            nc++;
        }
    }
    s.col_off[q.k] = nc;
    // 32-byte vector stores need 32-byte aligned columns
    for (int i = 0; i < nc; i++) vec &= ((uintptr_t)s.dst[i] & 31) == 0;
    s.vec = vec;
    s.A = A;
    s.err = q.ctx().err;
    return true;
}

gj_status tri_desummarize(QueryState &q, uint64_t row0, uint64_t nrows, void *const *out_cols,
                          uint32_t *const *rowid_cols, uint64_t *n_out);

gj_status cyc_desummarize(QueryState &q, uint64_t row0, uint64_t nrows, void *const *out_cols,
                          uint32_t *const *rowid_cols, uint64_t *n_out);

// wait: the rows are in place and the device error word checked on return;
// without it (the server, for queries over a join tree) both are the caller's.
gj_status desummarize(QueryState &q, uint64_t row0, uint64_t nrows, void *const *out_cols,
                      uint32_t *const *rowid_cols, uint64_t *n_out, bool wait) {
    if (q.tri) return tri_desummarize(q, row0, nrows, out_cols, rowid_cols, n_out);
    if (q.cyc) return cyc_desummarize(q, row0, nrows, out_cols, rowid_cols, n_out);
    Ctx &c = q.ctx();
    *n_out = 0;
    if (!q.summarized) return GJ_ERR_STATE;
    if (q.overflow) return GJ_ERR_OVERFLOW;
    if (row0 >= q.total || nrows == 0) return GJ_OK;
    uint64_t n = std::min<uint64_t>(nrows, q.total - row0);
    if (n > 0x7fffffffull) return GJ_ERR_INVALID;
    if ((int)q.var_rel.size() > MAXV || (int)q.col_rel.size() > MAXP) return GJ_ERR_INVALID;
    if (!out_cols) return GJ_ERR_INVALID;
    Frontier f;
    if (c.prof) cudaEventRecord(c.event(true), c.stream);
    // with two or more relations the last expansion level writes the emit
    // kernel's tile map itself
    TileMap tm{};
    if (q.k >= 2 && q.k <= 8) {
        tm.tile_rows = (int64_t)EMIT_DT * c.emit_rpt;
        tm.tiles = ceil_div((int64_t)n, tm.tile_rows);
        if (dalloc(c, &tm.tile_first, tm.tiles + 1) != cudaSuccess) return GJ_ERR_OOM;
    }
    cudaError_t e = expand(q, row0, row0 + n, q.k, false, f, tm.tile_first ? &tm : nullptr);
    if (c.prof) cudaEventRecord(c.event(true), c.stream);
    if (e != cudaSuccess) {
        dfree(c, tm.tile_first);
        return e == cudaErrorMemoryAllocation ? GJ_ERR_OOM : GJ_ERR_CUDA;
    }
    uint64_t width = 0;
    for (int v = 0; v < (int)q.var_rel.size(); v++) width += 4;
    for (size_t p = 0; p < q.col_rel.size(); p++) width += q.r[q.col_rel[p]].R->pw[q.col_pay[p]];
    if (q.k > 8 && c.prof) cudaEventRecord(c.event(), c.stream);
    if (q.k <= 8) {
        Emit4Spec s{};
        std::vector<const uint32_t *> grp(q.k);
        for (int j = 0; j < q.k; j++) grp[j] = f.grp[q.pos[j]];
        make_emit_spec(q, out_cols, rowid_cols, grp.data(), f.A, s);
        e = launch_emit(c, q.k, s, f.F_dev, row0, (int64_t)n, tm.tile_first);
    } else {
        EmitSpec s{};
        s.k = q.k;
        for (int j = 0; j < q.k; j++) {
            s.preidx[j] = q.pos[j];
            s.gstart[j] = q.r[j].F->gstart;
            s.perm[j] = q.r[j].F->perm;
            s.rid_out[j] = rowid_cols ? rowid_cols[j] : nullptr;
            s.grp[j] = f.grp[j];
        }
        s.nv = (int)q.var_rel.size();
        for (int v = 0; v < s.nv; v++) {
            const QRel &t = q.r[q.var_rel[v]];
            s.vkey[v] = t.F->key(q.var_col[v]);
            s.vrel[v] = q.var_rel[v];
            s.vout[v] = (int32_t *)out_cols[v];
        }
        s.np = (int)q.col_rel.size();
        for (int p = 0; p < s.np; p++) {
            const QRel &t = q.r[q.col_rel[p]];
            s.pay[p] = t.F->pay[q.col_pay[p]];
            s.prel[p] = q.col_rel[p];
            s.pw[p] = t.R->pw[q.col_pay[p]];
            s.pout[p] = out_cols[s.nv + p];
        }
        s.A = f.A;
        s.err = c.err;
        k_emit<<<(unsigned)ceil_div((int64_t)n, EMIT_TILE), DT, 0, c.stream>>>(s, f.F_dev, row0, (int64_t)n); c.launches++;
        e = cudaGetLastError();
    }
    if (c.prof) {
        cudaEventRecord(c.event(), c.stream);
        c.emit_launches++;
        c.emit_rows += n;
        c.emit_bytes += n * width;
    }
    frontier_free(c, f);
    dfree(c, tm.tile_first);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? GJ_ERR_OOM : GJ_ERR_CUDA;
    if (wait) {
        const gj_status st = check_device_error(c);
        if (st != GJ_OK) return st;
    }
    *n_out = n;
    return GJ_OK;
}

gj_status level_runs(QueryState &q, int level, uint64_t row0, uint64_t nrows, int32_t *val,
                     uint64_t *freq, uint64_t *off, uint64_t cap, uint64_t *n_out) {
    Ctx &c = q.ctx();
    *n_out = 0;
    if (q.tri || q.cyc) return GJ_ERR_INVALID;   // a cyclic join's summary is its block list
    if (!q.summarized) return GJ_ERR_STATE;
    if (q.overflow) return GJ_ERR_OVERFLOW;
    if (level < 0 || level >= (int)q.var_rel.size()) return GJ_ERR_INVALID;
    if (row0 >= q.total || nrows == 0) return GJ_OK;
    uint64_t n = std::min<uint64_t>(nrows, q.total - row0);
    if (n > 0x7fffffffull) return GJ_ERR_INVALID;
    const int tpos = q.var_rel[level];
    const QRel &t = q.r[tpos];
    const int j = q.pos[tpos];
    Frontier f;
    cudaError_t e = expand(q, row0, row0 + n, j + 1, true, f);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? GJ_ERR_OOM : GJ_ERR_CUDA;
    LevelSpec s{};
    s.A = f.A;
    s.lh = f.lh;
    s.unit = f.unit;
    s.lgid = t.lgid;
    s.loff = t.loff;
    s.lw = t.lw;
    s.seg_id = t.parent >= 0 ? t.seg_id : nullptr;
    s.lseg_first = t.lseg_first;
    s.L_dev = t.L_dev;
    int m = -1;
    for (size_t i = 0; i < t.new_cols.size(); i++)
        if (t.new_cols[i] == q.var_col[level]) m = (int)i;
    s.nprefix = m + 1;
    s.last = (m == (int)t.new_cols.size() - 1);
    for (int i = 0; i <= m; i++) s.pcol[i] = t.F->key(t.new_cols[i]);
    s.vcol = t.F->key(q.var_col[level]);
    // the run count goes into the word after the error word, so that one
    // readback brings both
    uint32_t *runs = c.err + 1, *idx = (uint32_t *)f.spare;
    const int sgrid = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(f.cap, EC_TILE), c.num_sms * 8));
    k_level_scan<<<sgrid, DT, 0, c.stream>>>(s, f.F_dev, row0, (uint32_t *)(f.state + 1), f.state + 2, idx, runs,
                                             c.err); c.launches++;
    k_level_write<<<grid_for(c, f.cap), DT, 0, c.stream>>>(s, f.F_dev, idx, runs, cap, val, freq, off); c.launches++;
    e = cudaGetLastError();
    uint32_t h[2] = {0, 0};
    if (e == cudaSuccess) e = readback(c, c.err, h, 8);
    frontier_free(c, f);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? GJ_ERR_OOM : GJ_ERR_CUDA;
    if (h[0]) {
        cudaMemsetAsync(c.err, 0, 4, c.stream);
        return h[0] & ERRF_TIMEOUT ? GJ_ERR_TIMEOUT : GJ_ERR_CUDA;
    }
    *n_out = h[1];
    return h[1] > cap ? GJ_ERR_CAPACITY : GJ_OK;
}

}  // namespace gj

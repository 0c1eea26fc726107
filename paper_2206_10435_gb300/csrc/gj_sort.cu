// gj_sort.cu -- stable LSD radix sort of (uint64 key, uint32 value) pairs.
//
// Used by factor construction to order a relation's rows by their packed
// join-key tuple (Section 3.2: the frequency table is the run-length form of
// the sorted rows).  8-bit digits, one "onesweep" launch per digit:
//
//   * one upfront pass reads every key once and builds the 256-bin
//     histogram of every digit in shared memory;
//   * per digit, each CTA takes the next tile id from a global counter,
//     ranks its 4096 keys with a warp-level multi-split (per-warp bins, no
//     atomics), publishes its per-digit counts,
//     finds each digit's global offset by decoupled lookback over the
//     preceding tiles (bounded polls, ERRF_TIMEOUT on expiry), stages the
//     tile in shared memory in digit order and scatters it so that
//     consecutive threads write consecutive addresses of a bucket.  The
//     bucket bases are scanned from the histogram by every CTA (256 values).
//
// A pass is bound by its instructions, not by DRAM (17% of it): whole tiles
// run without bounds checks, a lane reads its digit's bin and the last peer
// writes it back (no leader search, no shuffle), and the scatter reads one
// word per key.  1e7 words: 182 -> 144 issued instructions per 32 keys and
// 92 -> 72 us a pass, 68 with the matches below.
//
// Stable: ranks follow (tile, warp, item, lane) order, which is input order.
#include <algorithm>

#include "gj_internal.cuh"

namespace gj {
namespace {

constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_ITEMS = 16;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;       // 4096 keys
constexpr int RS_RADIX = 256;
constexpr int RS_MAX_PASSES = 8;
static_assert(RS_TILE == RADIX_SORT_TILE && RS_RADIX == RADIX_SORT_BINS &&
                  RS_MAX_PASSES == RADIX_SORT_MAX_PASSES,
              "the sort's tile layout is exported through gj_internal.cuh");
constexpr uint64_t ST_AGG = 1ull << 62, ST_PREFIX = 2ull << 62, ST_MASK = (1ull << 62) - 1;
// predecessors whose status a tile reads per round of its lookback (1e7 rows'
// factor: 2 946 us, 4 966, 8 990, 16 1031 -- more reads than a wait saves)
constexpr int RS_LOOKBACK = 2;
// every RS_MATCH-th item finds its peers by a match instead of ballots: the
// match unit and the ALUs then share the ranking (1e7 rows' factor: 842 us
// with ballots alone, 877 with matches alone, 820 with 2 or 3, 819 with 4)
constexpr int RS_MATCH = 4;
// resident CTAs per SM the keys-only kernel is compiled for
constexpr int RS_KEYS_CTAS = 4;

// Digits of eight words per thread and round, their loads issued together,
// column by column; the digits are unrolled (PASSES of them), so that each
// costs a field extract and one shared-memory atomic.  With a loop over the
// passes and all eight possible columns tested per word, 1e7 rows of two
// columns and five digits issued 171 instructions per 32 rows and took 72 us;
// 28 now (3e7 rows, one column, three digits: 191 -> 41).
constexpr int DH_ROWS = 8;

template <bool PACK, int PASSES>
__global__ void __launch_bounds__(RS_THREADS)
k_digit_hist(const uint64_t *__restrict__ keys, PackSrc ps, int64_t n, int lo_bit, uint32_t *hist) {
    __shared__ uint32_t sh[PASSES * RS_RADIX];
    for (int i = threadIdx.x; i < PASSES * RS_RADIX; i += RS_THREADS) sh[i] = 0;
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * RS_THREADS * DH_ROWS;
    for (int64_t b = (int64_t)blockIdx.x * RS_THREADS * DH_ROWS + threadIdx.x; b < n; b += step) {
        uint64_t k[DH_ROWS];
        if (PACK) {
#pragma unroll
            for (int u = 0; u < DH_ROWS; u++) k[u] = ps.row_bits ? (uint64_t)(b + u * RS_THREADS) : 0ull;
            for (int c = 0; c < ps.ncol; c++) {
                if (ps.shift[c] >= 64) continue;
                const int32_t *col = ps.col[c] + b;
                const uint32_t mn = (uint32_t)ps.mn[c];
                const int s = ps.shift[c];
                uint32_t x[DH_ROWS];
#pragma unroll
                for (int u = 0; u < DH_ROWS; u++)
                    x[u] = b + u * RS_THREADS < n ? (uint32_t)__ldg(col + u * RS_THREADS) : mn;
#pragma unroll
                for (int u = 0; u < DH_ROWS; u++) k[u] |= (uint64_t)(x[u] - mn) << s;
            }
        } else {
#pragma unroll
            for (int u = 0; u < DH_ROWS; u++)
                k[u] = b + u * RS_THREADS < n ? __ldg((const unsigned long long *)keys + b + u * RS_THREADS) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < DH_ROWS; u++) {
            if (b + u * RS_THREADS >= n) break;
            const uint64_t x = k[u] >> lo_bit;
#pragma unroll
            for (int p = 0; p < PASSES; p++)
                atomicAdd(sh + p * RS_RADIX + ((uint32_t)(x >> (8 * p)) & 0xffu), 1u);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < PASSES * RS_RADIX; i += RS_THREADS) {
        const uint32_t v = sh[i];
        if (v) atomicAdd(&hist[i], v);
    }
}

template <bool PACK>
void launch_hist(int passes, int grid, cudaStream_t st, const uint64_t *keys, const PackSrc &ps, int64_t n, int lo_bit,
                 uint32_t *hist) {
    switch (passes) {
        case 1: k_digit_hist<PACK, 1><<<grid, RS_THREADS, 0, st>>>(keys, ps, n, lo_bit, hist); break;
        case 2: k_digit_hist<PACK, 2><<<grid, RS_THREADS, 0, st>>>(keys, ps, n, lo_bit, hist); break;
        case 3: k_digit_hist<PACK, 3><<<grid, RS_THREADS, 0, st>>>(keys, ps, n, lo_bit, hist); break;
        case 4: k_digit_hist<PACK, 4><<<grid, RS_THREADS, 0, st>>>(keys, ps, n, lo_bit, hist); break;
        case 5: k_digit_hist<PACK, 5><<<grid, RS_THREADS, 0, st>>>(keys, ps, n, lo_bit, hist); break;
        case 6: k_digit_hist<PACK, 6><<<grid, RS_THREADS, 0, st>>>(keys, ps, n, lo_bit, hist); break;
        case 7: k_digit_hist<PACK, 7><<<grid, RS_THREADS, 0, st>>>(keys, ps, n, lo_bit, hist); break;
        default: k_digit_hist<PACK, 8><<<grid, RS_THREADS, 0, st>>>(keys, ps, n, lo_bit, hist); break;
    }
}

__device__ __forceinline__ unsigned long long ld_status(const unsigned long long *q) {
    return *(const volatile unsigned long long *)q;
}

// keys[i] = pack(i), vals[i] = i: a packed sort with nothing to order
__global__ void k_pack_words(PackSrc ps, int64_t n, uint64_t *__restrict__ keys, uint32_t *__restrict__ vals) {
    for (int64_t i = (int64_t)blockIdx.x * RS_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * RS_THREADS) {
        keys[i] = pack_word(ps, i);
        if (vals) vals[i] = (uint32_t)i;
    }
}

// One tile of a pass.  FULL: every position holds a key.
template <bool VALS, bool PACK, bool FULL>
__device__ __forceinline__ void
onesweep_tile(const uint64_t *__restrict__ kin, const PackSrc &ps, const uint32_t *__restrict__ vin,
              uint64_t *__restrict__ kout, uint32_t *__restrict__ vout, int64_t base, int tile_n, uint32_t tile,
              int shift, uint32_t count, unsigned long long *__restrict__ status, uint32_t *err,
              uint64_t *s_keys, uint32_t *s_vals, uint32_t *s_whist, uint32_t *s_dst, uint32_t *s_sum) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w0 = warp * (RS_ITEMS * 32) + lane;   // item i of this thread: position w0 + 32 i
    uint64_t k[RS_ITEMS];
    uint32_t v[RS_ITEMS];
    if (PACK) {
        // pass 0 of a packed sort builds the words from the key columns; per
        // column, the thread's 16 loads are issued together
#pragma unroll
        for (int i = 0; i < RS_ITEMS; i++) k[i] = ps.row_bits ? (uint64_t)(base + w0 + 32 * i) : 0ull;
        for (int c = 0; c < ps.ncol; c++) {
            if (ps.shift[c] >= 64) continue;
            const int32_t *col = ps.col[c] + base + w0;
            const uint32_t mn = (uint32_t)ps.mn[c];
            const int sh = ps.shift[c];
            uint32_t x[RS_ITEMS];
#pragma unroll
            for (int i = 0; i < RS_ITEMS; i++)
                x[i] = FULL || w0 + 32 * i < tile_n ? (uint32_t)__ldg(col + 32 * i) : mn;
#pragma unroll
            for (int i = 0; i < RS_ITEMS; i++) k[i] |= (uint64_t)(x[i] - mn) << sh;
        }
#pragma unroll
        for (int i = 0; i < RS_ITEMS; i++) v[i] = (uint32_t)(base + w0 + 32 * i);
    } else {
#pragma unroll
        for (int i = 0; i < RS_ITEMS; i++) {
            const bool in = FULL || w0 + 32 * i < tile_n;
            k[i] = in ? kin[base + w0 + 32 * i] : 0ull;
            v[i] = VALS && in ? vin[base + w0 + 32 * i] : 0u;
        }
    }
    // rank of every key among its warp's keys of the same digit, in order:
    // the peers of an item by one ballot per digit bit; every peer reads the
    // digit's count so far, the last one writes it back
    const uint32_t lt = (1u << lane) - 1u, gt = ~lt << 1;
    uint32_t *wh = s_whist + warp * RS_RADIX;
    uint32_t rank[RS_ITEMS];                        // digit << 16 | rank
#pragma unroll
    for (int i = 0; i < RS_ITEMS; i++) {
        const bool in = FULL || w0 + 32 * i < tile_n;
        const uint32_t d = (uint32_t)(k[i] >> shift) & 0xffu;
        uint32_t peers;
        if (i % RS_MATCH == 0) {
            peers = __match_any_sync(0xffffffffu, FULL || in ? d : 0x100u);
        } else {
            peers = FULL ? 0xffffffffu : __ballot_sync(0xffffffffu, in);
#pragma unroll
            for (int b = 0; b < 8; b++) {
                const bool bit = d & (1u << b);
                const uint32_t bal = __ballot_sync(0xffffffffu, bit);
                peers &= bit ? bal : ~bal;
            }
        }
        const uint32_t r = wh[d] + __popc(peers & lt);
        __syncwarp();
        if (in && (peers & gt) == 0) wh[d] = r + 1;
        __syncwarp();
        rank[i] = d << 16 | r;
    }
    __syncthreads();
    // per digit (thread d): the tile's count, published, then its prefix
    // over the preceding tiles
    const int d = tid;   // RS_THREADS == RS_RADIX
    uint32_t cnt = 0;
#pragma unroll
    for (int w = 0; w < RS_WARPS; w++) cnt += s_whist[w * RS_RADIX + d];
    unsigned long long *st = status + (size_t)tile * RS_RADIX + d;
    *(volatile unsigned long long *)st = (tile == 0 ? ST_PREFIX : ST_AGG) | cnt;
    // exclusive offsets over the digits, of the tile's counts and of the
    // whole input's (the bucket bases): a shuffle scan per warp of 32 digits,
    // then the totals of the preceding warps
    uint32_t x = cnt, y = count;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t a = __shfl_up_sync(0xffffffffu, x, off), b = __shfl_up_sync(0xffffffffu, y, off);
        if (lane >= off) { x += a; y += b; }
    }
    if (lane == 31) { s_sum[warp] = x; s_sum[RS_WARPS + warp] = y; }
    __syncthreads();
    uint32_t tile_off = x - cnt, bucket = y - count;
    for (int w = 0; w < warp; w++) { tile_off += s_sum[w]; bucket += s_sum[RS_WARPS + w]; }
    {
        uint32_t run = tile_off;
#pragma unroll
        for (int w = 0; w < RS_WARPS; w++) {
            const uint32_t mine = s_whist[w * RS_RADIX + d];
            s_whist[w * RS_RADIX + d] = run;
            run += mine;
        }
    }
    // look back RS_LOOKBACK predecessors per round (their status words are
    // read together, then folded nearest first; one that has published
    // nothing yet is polled, bounded, before the fold goes on)
    uint64_t excl = 0;
    if (tile != 0) {
        int64_t p = (int64_t)tile - 1;
        bool done = false;
        while (!done && p >= 0) {
            unsigned long long sv[RS_LOOKBACK];
#pragma unroll
            for (int j = 0; j < RS_LOOKBACK; j++)
                sv[j] = p - j >= 0 ? ld_status(status + (size_t)(p - j) * RS_RADIX + d)
                                   : (unsigned long long)ST_PREFIX;
#pragma unroll
            for (int j = 0; j < RS_LOOKBACK; j++) {
                if (!done) {
                    unsigned long long s = sv[j];
                    uint32_t spins = 0;
                    while ((s >> 62) == 0) {
                        if (++spins > SPIN_LIMIT) { raise_err(err, ERRF_TIMEOUT); s = ST_PREFIX; break; }
                        s = ld_status(status + (size_t)(p - j) * RS_RADIX + d);
                    }
                    excl += s & ST_MASK;
                    done = (s & ST_PREFIX) != 0;
                }
            }
            p -= RS_LOOKBACK;
        }
        *(volatile unsigned long long *)st = ST_PREFIX | (excl + cnt);
    }
    s_dst[d] = bucket + (uint32_t)excl - tile_off;   // + staged position = destination
    __syncthreads();
    // stage in digit order
#pragma unroll
    for (int i = 0; i < RS_ITEMS; i++) {
        if (FULL || w0 + 32 * i < tile_n) {
            const uint32_t pos = wh[rank[i] >> 16] + (rank[i] & 0xffffu);
            s_keys[pos] = k[i];
            if (VALS) s_vals[pos] = v[i];
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RS_ITEMS; i++) {
        const int p = i * RS_THREADS + tid;
        if (FULL || p < tile_n) {
            const uint64_t key = s_keys[p];
            const uint32_t dest = s_dst[(uint32_t)(key >> shift) & 0xffu] + (uint32_t)p;
            kout[dest] = key;
            if (VALS) vout[dest] = s_vals[p];
        }
    }
}

template <bool VALS, bool PACK>
__global__ void __launch_bounds__(RS_THREADS, VALS ? 3 : RS_KEYS_CTAS)
k_onesweep_t(const uint64_t *__restrict__ kin, PackSrc ps, const uint32_t *__restrict__ vin,
             uint64_t *__restrict__ kout, uint32_t *__restrict__ vout, int64_t n, int shift,
             const uint32_t *__restrict__ hist, uint32_t *tile_counter,
             unsigned long long *status, uint32_t *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *s_keys = (uint64_t *)smem;                              // RS_TILE
    uint32_t *s_vals = (uint32_t *)(s_keys + RS_TILE);                // RS_TILE (VALS only)
    uint32_t *s_whist = s_vals + (VALS ? RS_TILE : 0);                // RS_WARPS*RS_RADIX
    uint32_t *s_dst = s_whist + RS_WARPS * RS_RADIX;                  // RS_RADIX
    uint32_t *s_misc = s_dst + RS_RADIX;                              // 2*RS_WARPS + 1
    const int tid = threadIdx.x;
    if (tid == 0) s_misc[2 * RS_WARPS] = atomicAdd(tile_counter, 1u);
    for (int i = tid; i < RS_WARPS * RS_RADIX; i += RS_THREADS) s_whist[i] = 0;
    const uint32_t count = hist[tid];                                 // digit tid's keys, all tiles
    __syncthreads();
    const uint32_t tile = s_misc[2 * RS_WARPS];
    const int64_t base = (int64_t)tile * RS_TILE;
    if (n - base >= RS_TILE)
        onesweep_tile<VALS, PACK, true>(kin, ps, vin, kout, vout, base, RS_TILE, tile, shift, count, status, err,
                                        s_keys, s_vals, s_whist, s_dst, s_misc);
    else
        onesweep_tile<VALS, PACK, false>(kin, ps, vin, kout, vout, base, (int)(n - base), tile, shift, count, status,
                                         err, s_keys, s_vals, s_whist, s_dst, s_misc);
}

constexpr size_t rs_smem(bool vals) {
    return (size_t)RS_TILE * (vals ? 12 : 8) + (size_t)RS_WARPS * RS_RADIX * 4 + RS_RADIX * 4 + (2 * RS_WARPS + 1) * 4;
}

template <bool VALS, bool PACK>
cudaError_t onesweep_prepare(int device) {
    return set_max_shared_once<k_onesweep_t<VALS, PACK>>(device, rs_smem(VALS));
}

template <bool VALS, bool PACK>
cudaError_t onesweep(Ctx &c, const uint64_t *ka, const PackSrc &ps, const uint32_t *va, uint64_t *kb, uint32_t *vb,
                     int64_t n, int shift, const uint32_t *hist, uint32_t *counter, unsigned long long *status) {
    GJ_CUDA_TRY((onesweep_prepare<VALS, PACK>(c.device)));
    k_onesweep_t<VALS, PACK><<<(unsigned)ceil_div(n, RS_TILE), RS_THREADS, rs_smem(VALS), c.stream>>>(
        ka, ps, va, kb, vb, n, shift, hist, counter, status, c.err);
    c.launches++;
    return cudaGetLastError();
}

constexpr size_t HIST_WORDS = RS_MAX_PASSES * RS_RADIX + RS_MAX_PASSES;   // histograms, then tile counters

// The histogram and the passes of a sort (n > 1, passes > 0) on scratch that
// the caller gives: hist holds HIST_WORDS words, status one word per tile and
// digit; `cleared`: hist and every pass's status (consecutive) are zero, else
// they are cleared here, one pass's status at a time.
cudaError_t sort_passes(Ctx &c, const PackSrc *pack, uint64_t *ka, uint64_t *kb, uint32_t *va, uint32_t *vb,
                        int64_t n, int lo_bit, int passes, uint32_t *hist, unsigned long long *status, bool cleared,
                        uint64_t **kres, uint32_t **vres) {
    const size_t status_words = (size_t)ceil_div(n, RS_TILE) * RS_RADIX;
    uint32_t *counters = hist + RS_MAX_PASSES * RS_RADIX;
    if (!cleared) GJ_CUDA_TRY(cudaMemsetAsync(hist, 0, sizeof(uint32_t) * HIST_WORDS, c.stream));
    const PackSrc ps = pack ? *pack : PackSrc{};
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, RS_THREADS * 16), (int64_t)c.num_sms * 8));
    if (pack) launch_hist<true>(passes, grid, c.stream, nullptr, ps, n, lo_bit, hist);
    else launch_hist<false>(passes, grid, c.stream, ka, ps, n, lo_bit, hist);
    c.launches++;
    GJ_CUDA_TRY(cudaGetLastError());
    for (int p = 0; p < passes; p++) {
        unsigned long long *st = status + (cleared ? status_words * (size_t)p : 0);
        if (!cleared) GJ_CUDA_TRY(cudaMemsetAsync(st, 0, sizeof(unsigned long long) * status_words, c.stream));
        const int shift = lo_bit + 8 * p;
        const uint32_t *h = hist + p * RS_RADIX;
        // the first pass of a packed sort reads the columns and writes into
        // `kb`; later passes ping-pong
        cudaError_t e;
        if (va && p == 0 && pack) e = onesweep<true, true>(c, nullptr, ps, nullptr, kb, vb, n, shift, h, counters + p, st);
        else if (va) e = onesweep<true, false>(c, ka, ps, va, kb, vb, n, shift, h, counters + p, st);
        else if (p == 0 && pack) e = onesweep<false, true>(c, nullptr, ps, nullptr, kb, nullptr, n, shift, h, counters + p, st);
        else e = onesweep<false, false>(c, ka, ps, nullptr, kb, nullptr, n, shift, h, counters + p, st);
        GJ_CUDA_TRY(e);
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    *kres = ka;
    if (vres) *vres = va;
    return cudaSuccess;
}

// Up to this many tiles every pass has its own status words, cleared together
// with the histogram (64 MB at 8 passes); beyond, the clears are small next
// to the passes and share one pass's words.
constexpr int64_t SORT_CLEAR_TILES = 4096;

// sort_passes on scratch from the context
cudaError_t sort_alloc(Ctx &c, const PackSrc *pack, uint64_t *keys, uint64_t *alt, uint32_t *vals, uint32_t *valt,
                       int64_t n, int lo_bit, int passes, uint64_t **kres, uint32_t **vres) {
    const int64_t tiles = ceil_div(n, RS_TILE);
    const bool all = tiles <= SORT_CLEAR_TILES;
    const size_t hist_bytes = (sizeof(uint32_t) * HIST_WORDS + 255) & ~(size_t)255;
    const size_t status_bytes = sizeof(unsigned long long) * (size_t)tiles * RS_RADIX * (size_t)(all ? passes : 1);
    char *scratch = nullptr;
    Temps tmp(c);
    GJ_CUDA_TRY(tmp.alloc(&scratch, hist_bytes + status_bytes));
    if (all) GJ_CUDA_TRY(cudaMemsetAsync(scratch, 0, hist_bytes + status_bytes, c.stream));
    return sort_passes(c, pack, keys, alt, vals, valt, n, lo_bit, passes, (uint32_t *)scratch,
                       (unsigned long long *)(scratch + hist_bytes), all, kres, vres);
}

// the sorted result in the caller's own buffers
cudaError_t copy_back(Ctx &c, uint64_t *keys, uint64_t *kres, uint32_t *vals, uint32_t *vres, int64_t n) {
    if (kres == keys) return cudaSuccess;
    GJ_CUDA_TRY(cudaMemcpyAsync(keys, kres, sizeof(uint64_t) * n, cudaMemcpyDeviceToDevice, c.stream));
    if (vals) GJ_CUDA_TRY(cudaMemcpyAsync(vals, vres, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, c.stream));
    return cudaSuccess;
}

}  // namespace

cudaError_t radix_sort_u64_u32(Ctx &c, uint64_t *keys, uint32_t *vals, int64_t n, int bits) {
    if (n <= 1 || bits <= 0) return cudaSuccess;
    if (n > 0x7fffffffLL || bits > 64) return cudaErrorInvalidValue;
    uint64_t *k2 = nullptr, *kres = nullptr;
    uint32_t *v2 = nullptr, *vres = nullptr;
    Temps tmp(c);
    GJ_CUDA_TRY(tmp.alloc(&k2, n));
    GJ_CUDA_TRY(tmp.alloc(&v2, n));
    GJ_CUDA_TRY(sort_alloc(c, nullptr, keys, k2, vals, v2, n, 0, (bits + 7) / 8, &kres, &vres));
    return copy_back(c, keys, kres, vals, vres, n);
}

// Same sort with every scratch buffer supplied by the caller (no device
// allocation): k2/v2 hold n entries, hist 8*256 + 8 words, status
// status_tiles*256 words (status_tiles >= ceil(n / 4096)).
cudaError_t radix_sort_u64_u32_in(Ctx &c, uint64_t *keys, uint32_t *vals, int64_t n, int bits,
                                  uint64_t *k2, uint32_t *v2, uint32_t *hist,
                                  unsigned long long *status, int64_t status_tiles) {
    if (n <= 1 || bits <= 0) return cudaSuccess;
    if (n > 0x7fffffffLL || bits > 64) return cudaErrorInvalidValue;
    if (ceil_div(n, RS_TILE) > status_tiles) return cudaErrorInvalidValue;
    uint64_t *kres = nullptr;
    uint32_t *vres = nullptr;
    GJ_CUDA_TRY(sort_passes(c, nullptr, keys, k2, vals, v2, n, 0, (bits + 7) / 8, hist, status, false, &kres, &vres));
    return copy_back(c, keys, kres, vals, vres, n);
}

// Sets the keys-only sort kernel's shared-memory limit; call once before
// any capture of radix_sort_keys_u64_in.
cudaError_t radix_sort_keys_prepare(int device) { return onesweep_prepare<false, false>(device); }

// Keys-only sort with caller scratch (no allocation, capturable in a CUDA
// graph): k2 holds n keys, hist 8*256 + 8 words, status status_tiles*256
// words.  Accepts up to 2^32 - 1 keys.
cudaError_t radix_sort_keys_u64_in(Ctx &c, uint64_t *keys, int64_t n, int bits, uint64_t *k2,
                                   uint32_t *hist, unsigned long long *status,
                                   int64_t status_tiles) {
    if (n <= 1 || bits <= 0) return cudaSuccess;
    if (n > 0xffffffffLL || bits > 64) return cudaErrorInvalidValue;
    if (ceil_div(n, RS_TILE) > status_tiles) return cudaErrorInvalidValue;
    uint64_t *kres = nullptr;
    GJ_CUDA_TRY(sort_passes(c, nullptr, keys, k2, nullptr, nullptr, n, 0, (bits + 7) / 8, hist, status, false, &kres,
                            nullptr));
    return copy_back(c, keys, kres, nullptr, nullptr, n);
}

cudaError_t radix_sort_words(Ctx &c, const PackSrc *pack, uint64_t *keys, uint64_t *alt,
                             uint32_t *vals, uint32_t *valt, int64_t n, int lo_bit, int bits,
                             uint64_t **kres, uint32_t **vres) {
    *kres = keys;
    if (vres) *vres = vals;
    if (n > 0x7fffffffLL || bits < 0 || lo_bit < 0 || lo_bit + bits > 64) return cudaErrorInvalidValue;
    const int passes = (bits + 7) / 8;
    if (n == 0) return cudaSuccess;
    if (passes == 0 || n == 1) {
        // nothing to order: the words (and row ids) in input order
        if (pack) {
            const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, RS_THREADS), (int64_t)c.num_sms * 16));
            k_pack_words<<<grid, RS_THREADS, 0, c.stream>>>(*pack, n, keys, vals); c.launches++;
            GJ_CUDA_TRY(cudaGetLastError());
        }
        return cudaSuccess;
    }
    return sort_alloc(c, pack, keys, alt, vals, valt, n, lo_bit, passes, kres, vres);
}

}  // namespace gj

// gj_factor_small.cu -- factor construction of small relations, one CTA each.
//
// A relation of a few thousand rows spends its build on launches: key ranges,
// a readback, histogram, sort passes, group scan, a readback, the keys' move,
// each of a few microseconds and each on one or two CTAs.  Here one launch
// builds up to SF_BATCH relations, a CTA per relation with everything in
// shared memory and registers: the columns' ranges, the packed words (key over
// row id), their stable radix sort (8-bit digits; peers by ballots, per-warp
// bins), the groups with their starts and keys, and the payloads in group
// order.  The ranges and group counts of all relations come back in the one
// readback that the caller makes.  A key that does not fit a word beside the
// row id leaves only its ranges behind (the caller builds it another way).
//
// Bound by latency: a few barriers and shared-memory rounds per digit.  A join
// of three relations of 1000 rows: 68 -> 19 device operations, 0.46 -> 0.28 ms
// (this kernel 14 us); of 10^4 rows, host to host: 0.69 -> 0.50 ms (44 us).
// SF_MAX is what one CTA's shared memory and 64 registers a thread hold; the
// sort's CTAs would take over a little above it (its passes are 8 us each).
#include <algorithm>

#include "gj_factor_small.cuh"

namespace gj {
namespace {

constexpr int SF_THREADS = 1024;
constexpr int SF_WARPS = SF_THREADS / 32;
constexpr int SF_RADIX = 256;
constexpr int SF_BATCH = 16;

struct SfRel {
    int n, nk, nord, np;
    int order[MAX_KEYS];
    const int32_t *key[MAX_KEYS];
    const void *pay_in[MAX_PAYLOADS];
    void *pay_out[MAX_PAYLOADS];
    int pw[MAX_PAYLOADS];
    uint32_t *perm, *gstart;
    int32_t *gkey;
    int32_t *out;                  // [SF_OUT]: groups, whether built, the columns' ranges
};
struct SfSpec {
    SfRel r[SF_BATCH];
};

__device__ __forceinline__ int sf_bits(uint32_t range) { return range == 0 ? 0 : 32 - __clz((int)range); }

// ITEMS rows per thread.  Row item i of a thread: warp * 32 ITEMS + 32 i + lane.
template <int ITEMS>
__global__ void __launch_bounds__(SF_THREADS, 1) k_small_factor(const __grid_constant__ SfSpec S) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *s_keys = (uint64_t *)smem;                              // [ITEMS * SF_THREADS]
    uint16_t *s_hist = (uint16_t *)(s_keys + ITEMS * SF_THREADS);     // [SF_WARPS][SF_RADIX]
    __shared__ int s_mn[MAX_KEYS], s_mx[MAX_KEYS];
    __shared__ uint32_t s_sum[SF_WARPS], s_cnt[ITEMS * SF_WARPS];
    const SfRel &r = S.r[blockIdx.x];
    const int n = r.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w0 = warp * (32 * ITEMS) + lane;
    const uint32_t lt = (1u << lane) - 1u, gt = ~lt << 1;
    if (tid < MAX_KEYS) {
        s_mn[tid] = INT32_MAX;
        s_mx[tid] = INT32_MIN;
    }
    __syncthreads();
    for (int c = 0; c < r.nk; c++) {
        int lo = INT32_MAX, hi = INT32_MIN;
#pragma unroll
        for (int i = 0; i < ITEMS; i++)
            if (w0 + 32 * i < n) {
                const int v = __ldg(r.key[c] + w0 + 32 * i);
                lo = min(lo, v);
                hi = max(hi, v);
            }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0 && lo <= hi) {
            atomicMin(&s_mn[c], lo);
            atomicMax(&s_mx[c], hi);
        }
    }
    __syncthreads();
    if (tid < r.nk) {
        r.out[2 + 2 * tid] = s_mn[tid];
        r.out[3 + 2 * tid] = s_mx[tid];
    }
    const int row_bits = sf_bits((uint32_t)(n - 1));
    int kbits = 0;
    for (int o = 0; o < r.nord; o++) {
        const int c = r.order[o];
        kbits += sf_bits((uint32_t)s_mx[c] - (uint32_t)s_mn[c]);
    }
    if (kbits + row_bits > 64) {
        if (tid == 0) {
            r.out[0] = 0;
            r.out[1] = 0;
        }
        return;
    }
    // words: the row id under the key, the order's last column lowest
    uint64_t k[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; i++) k[i] = (uint64_t)(w0 + 32 * i);
    for (int o = r.nord - 1, shift = row_bits; o >= 0; o--) {
        const int c = r.order[o];
        const uint32_t mn = (uint32_t)s_mn[c];
        const int b = sf_bits((uint32_t)s_mx[c] - mn);
        if (b == 0) continue;
#pragma unroll
        for (int i = 0; i < ITEMS; i++)
            if (w0 + 32 * i < n) k[i] |= (uint64_t)((uint32_t)__ldg(r.key[c] + w0 + 32 * i) - mn) << shift;
        shift += b;
    }
    if (kbits == 0) {
#pragma unroll
        for (int i = 0; i < ITEMS; i++) s_keys[w0 + 32 * i] = k[i];
        __syncthreads();
    }
    uint16_t *wh = s_hist + warp * SF_RADIX;
    for (int bit = row_bits; bit < row_bits + kbits; bit += 8) {
        for (int i = tid; i < SF_WARPS * SF_RADIX / 2; i += SF_THREADS) ((uint32_t *)s_hist)[i] = 0;
        __syncthreads();
        // rank among the warp's keys of the same digit, two to a word
        uint32_t rank[(ITEMS + 1) / 2];
#pragma unroll
        for (int i = 0; i < ITEMS; i++) {
            const bool in = w0 + 32 * i < n;
            const uint32_t d = (uint32_t)(k[i] >> bit) & 0xffu;
            uint32_t peers = __ballot_sync(0xffffffffu, in);
#pragma unroll
            for (int b = 0; b < 8; b++) {
                const bool on = d & (1u << b);
                const uint32_t bal = __ballot_sync(0xffffffffu, on);
                peers &= on ? bal : ~bal;
            }
            const uint32_t x = wh[d] + __popc(peers & lt);
            __syncwarp();
            if (in && (peers & gt) == 0) wh[d] = (uint16_t)(x + 1);
            __syncwarp();
            if (i & 1) rank[i / 2] |= x << 16;
            else rank[i / 2] = x;
        }
        __syncthreads();
        uint32_t cnt = 0, x = 0;
        if (tid < SF_RADIX) {
#pragma unroll 8
            for (int w = 0; w < SF_WARPS; w++) cnt += s_hist[w * SF_RADIX + tid];
            x = cnt;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
                if (lane >= d) x += y;
            }
            if (lane == 31) s_sum[warp] = x;
        }
        __syncthreads();
        if (tid < SF_RADIX) {
            uint32_t at = x - cnt;
            for (int w = 0; w < warp; w++) at += s_sum[w];
#pragma unroll 8
            for (int w = 0; w < SF_WARPS; w++) {
                const uint32_t c = s_hist[w * SF_RADIX + tid];
                s_hist[w * SF_RADIX + tid] = (uint16_t)at;
                at += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < ITEMS; i++)
            if (w0 + 32 * i < n) {
                const uint32_t d = (uint32_t)(k[i] >> bit) & 0xffu;
                s_keys[wh[d] + ((i & 1) ? rank[i / 2] >> 16 : rank[i / 2] & 0xffffu)] = k[i];
            }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < ITEMS; i++)
            if (w0 + 32 * i < n) k[i] = s_keys[w0 + 32 * i];
    }
    // group heads, row e = i * SF_THREADS + tid, and their numbers in row order
    uint32_t hb[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
        const int e = i * SF_THREADS + tid;
        const bool h = e < n && (e == 0 || (s_keys[e] >> row_bits) != (s_keys[e - 1] >> row_bits));
        hb[i] = __ballot_sync(0xffffffffu, h);
        if (lane == 0) s_cnt[i * SF_WARPS + warp] = __popc(hb[i]);
    }
    __syncthreads();
    if (warp < ITEMS) {
        const uint32_t c = s_cnt[warp * SF_WARPS + lane];
        uint32_t x = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        s_cnt[warp * SF_WARPS + lane] = x - c;
        if (lane == 31) s_sum[warp] = x;
    }
    __syncthreads();
    uint32_t G = 0;
    for (int i = 0; i < ITEMS; i++) G += s_sum[i];
    const uint32_t rmask = row_bits ? (uint32_t)((1ull << row_bits) - 1) : 0u;
    uint32_t first = 0;
#pragma unroll 1
    for (int i = 0; i < ITEMS; i++) {
        const int e = i * SF_THREADS + tid;
        if (e < n) {
            const uint64_t word = s_keys[e];
            const uint32_t row = (uint32_t)word & rmask;
            r.perm[e] = row;
            for (int p = 0; p < r.np; p++) {
                if (r.pw[p] == 8)
                    ((unsigned long long *)r.pay_out[p])[e] = __ldg((const unsigned long long *)r.pay_in[p] + row);
                else
                    ((unsigned int *)r.pay_out[p])[e] = __ldg((const unsigned int *)r.pay_in[p] + row);
            }
            uint32_t heads = 0;
#pragma unroll
            for (int j = 0; j < ITEMS; j++)
                if (j == i) heads = hb[j];
            if ((heads >> lane) & 1u) {
                const uint32_t g = first + s_cnt[i * SF_WARPS + warp] + __popc(heads & lt);
                r.gstart[g] = (uint32_t)e;
                for (int c = 0; c < r.nk; c++) r.gkey[(int64_t)c * G + g] = __ldg(r.key[c] + row);
            }
        }
        first += s_sum[i];
    }
    if (tid == 0) {
        r.gstart[G] = (uint32_t)n;
        r.out[0] = (int32_t)G;
        r.out[1] = 1;
    }
}

template <int ITEMS>
cudaError_t launch_small(Ctx &c, const SfSpec &s, int count) {
    constexpr size_t smem = (size_t)ITEMS * SF_THREADS * 8 + (size_t)SF_WARPS * SF_RADIX * 2;
    GJ_CUDA_TRY(set_max_shared_once<k_small_factor<ITEMS>>(c.device, smem));
    k_small_factor<ITEMS><<<count, SF_THREADS, smem, c.stream>>>(s);
    c.launches++;
    return cudaGetLastError();
}

}  // namespace

cudaError_t small_factors(Ctx &c, const std::vector<SmallFactor> &f) {
    // relations of few rows per thread together, the larger ones apart
    for (int big = 0; big < 2; big++) {
        SfSpec s{};
        int m = 0;
        for (size_t i = 0; i < f.size(); i++) {
            const Relation &R = *f[i].R;
            Factor &F = *f[i].F;
            if ((R.n > 4 * SF_THREADS) == (big == 1)) {
                SfRel &x = s.r[m++];
                x.n = (int)R.n;
                x.nk = R.nk;
                x.nord = (int)F.order.size();
                x.np = R.np;
                for (int o = 0; o < x.nord; o++) x.order[o] = F.order[o];
                for (int k = 0; k < R.nk; k++) x.key[k] = R.key[k];
                for (int p = 0; p < R.np; p++) {
                    x.pay_in[p] = R.pay[p];
                    x.pay_out[p] = F.pay[p];
                    x.pw[p] = R.pw[p];
                }
                x.perm = F.perm;
                x.gstart = F.gstart;
                x.gkey = F.gkey;
                x.out = f[i].out;
            }
            if (m == SF_BATCH || (m > 0 && i + 1 == f.size())) {
                GJ_CUDA_TRY(big ? launch_small<SF_MAX / SF_THREADS>(c, s, m) : launch_small<4>(c, s, m));
                m = 0;
            }
        }
    }
    return cudaSuccess;
}

}  // namespace gj

// gj_scan.cu -- single-pass exclusive prefix sums with decoupled lookback.
//
// One launch per scan: every CTA takes the next tile id from a global
// counter (so a tile only ever waits on tiles that are already running),
// scans the tile, publishes the tile's aggregate, looks back over its
// predecessors' published aggregates/prefixes to find its carry-in, and
// publishes its inclusive prefix.  Polls of a predecessor's flag are bounded
// by SPIN_LIMIT; on expiry the kernel records ERRF_TIMEOUT and carries on,
// so a stuck predecessor can never hang the GPU.
#include <algorithm>

#include "gj_lookback.cuh"

namespace gj {
namespace {

constexpr int SCAN_THREADS = 256;

// The tile's carry-in and every warp's sum before it: `sum` is the warp's
// total (the same in every lane), returned is the sum of everything before
// the warp.
template <class T, class Op, int THREADS>
__device__ __forceinline__ T warp_carry(T sum, uint32_t tile, bool last, typename TileStatus<T>::W *status, T *total,
                                        T *s_warp, T *s_carry, uint32_t *err) {
    Op op;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) s_warp[warp] = sum;
    __syncthreads();
    T before = T(0);
    for (int w = 0; w < warp; w++) before = op(before, s_warp[w]);
    if (warp == THREADS / 32 - 1) {
        const T agg = op(before, sum);
        const T carry = warp_lookback<T, Op>(status, tile, agg, lane, err);
        if (lane == 0) {
            *s_carry = carry;
            if (last && total) *total = op(carry, agg);
        }
    }
    __syncthreads();
    return op(*s_carry, before);
}

// 32-bit sums of words or of byte flags; a warp scans 512 consecutive
// elements, 32 at a time.
constexpr int U32_ITEMS = 16;
static_assert(SCAN_THREADS * U32_ITEMS == SCAN_U32_TILE, "the 32-bit scan tile is exported through gj_internal.cuh");

__global__ void __launch_bounds__(SCAN_THREADS)
k_scan_u32(const uint32_t *__restrict__ in, const uint8_t *__restrict__ flags, uint32_t *__restrict__ out, int64_t n,
           uint32_t *tile_counter, unsigned long long *status, uint32_t *total, uint32_t *err) {
    __shared__ uint32_t s_warp[SCAN_THREADS / 32], s_carry, s_tile;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_tile = atomicAdd(tile_counter, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const int64_t base = (int64_t)tile * SCAN_U32_TILE;
    if (base >= n) return;
    const int64_t w0 = base + warp * (32 * U32_ITEMS) + lane;
    uint32_t x[U32_ITEMS];
#pragma unroll
    for (int i = 0; i < U32_ITEMS; i++) {
        const int64_t e = w0 + 32 * i;
        x[i] = e < n ? (in ? in[e] : (uint32_t)(flags[e] != 0)) : 0u;
    }
    uint32_t run = 0;
#pragma unroll
    for (int i = 0; i < U32_ITEMS; i++) {
        uint32_t v = x[i];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, v, d);
            if (lane >= d) v += y;
        }
        x[i] = run + v - x[i];                              // exclusive in the warp
        run += __shfl_sync(0xffffffffu, v, 31);
    }
    const uint32_t carry = warp_carry<uint32_t, AddU32, SCAN_THREADS>(run, tile, base + SCAN_U32_TILE >= n, status, total, s_warp,
                                                        &s_carry, err);
#pragma unroll
    for (int i = 0; i < U32_ITEMS; i++)
        if (w0 + 32 * i < n) out[w0 + 32 * i] = carry + x[i];
}

// Saturating 64-bit sums; a lane takes two consecutive elements with one
// 16-byte access, a warp 64 at a time, in registers throughout.  3.6e7
// elements: 142 us (4.1 TB/s); 178 with tiles of 2048 elements (the prefixes
// travel along the tiles at about 100 a microsecond) and 152 with 8192 (128
// registers a thread, half the threads in flight).
constexpr int U64_PAIRS = 8;
constexpr int U64_THREADS = 256;
constexpr int U64_TILE = U64_THREADS * U64_PAIRS * 2;

__global__ void __launch_bounds__(U64_THREADS)
k_scan_u64_sat(const ulonglong2 *__restrict__ in, ulonglong2 *__restrict__ out, int64_t n, uint32_t *tile_counter,
               ulonglong2 *status, uint64_t *total, uint32_t *err) {
    __shared__ uint64_t s_warp[U64_THREADS / 32], s_carry;
    __shared__ uint32_t s_tile;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_tile = atomicAdd(tile_counter, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const int64_t base = (int64_t)tile * U64_TILE;
    if (base >= n) return;
    const int64_t p0 = base / 2 + warp * (32 * U64_PAIRS) + lane;    // pair i of this lane: p0 + 32 i
    ulonglong2 x[U64_PAIRS];
#pragma unroll
    for (int i = 0; i < U64_PAIRS; i++) {
        const int64_t p = p0 + 32 * i;
        x[i] = make_ulonglong2(0, 0);
        if (2 * p + 1 < n) x[i] = in[p];
        else if (2 * p < n) x[i].x = ((const unsigned long long *)in)[2 * p];
    }
    uint64_t run = 0;
#pragma unroll
    for (int i = 0; i < U64_PAIRS; i++) {
        uint64_t v = sat_add(x[i].x, x[i].y);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, v, d);
            if (lane >= d) v = sat_add(y, v);
        }
        uint64_t ex = __shfl_up_sync(0xffffffffu, v, 1);
        ex = lane == 0 ? run : sat_add(run, ex);
        x[i].y = sat_add(ex, x[i].x);                       // exclusive in the warp
        x[i].x = ex;
        run = sat_add(run, __shfl_sync(0xffffffffu, v, 31));
    }
    const uint64_t carry = warp_carry<uint64_t, SatAddU64, U64_THREADS>(run, tile, base + U64_TILE >= n, status, total, s_warp,
                                                           &s_carry, err);
#pragma unroll
    for (int i = 0; i < U64_PAIRS; i++) {
        const int64_t p = p0 + 32 * i;
        const ulonglong2 y = make_ulonglong2(sat_add(carry, x[i].x), sat_add(carry, x[i].y));
        if (2 * p + 1 < n) out[p] = y;
        else if (2 * p < n) ((unsigned long long *)out)[2 * p] = y.x;
    }
}

}  // namespace

size_t scan_u32_state_bytes(int64_t n) { return scan_u32_state_bytes_for(n); }

// scan_u32 with the lookback state in caller memory (no device allocation):
// state must hold scan_u32_state_bytes(n) bytes.
cudaError_t scan_u32_in(Ctx &c, const uint32_t *in, const uint8_t *flags, uint32_t *out,
                        int64_t n, uint32_t *total_dev, void *state_mem, size_t state_bytes) {
    if (n <= 0) {
        if (total_dev) GJ_CUDA_TRY(cudaMemsetAsync(total_dev, 0, sizeof(uint32_t), c.stream));
        return cudaSuccess;
    }
    if (state_bytes < scan_u32_state_bytes(n)) return cudaErrorInvalidValue;
    const int64_t tiles = ceil_div(n, SCAN_U32_TILE);
    if (tiles > 0x7fffffff) return cudaErrorInvalidValue;
    // the tile counter, then the tiles' status words
    GJ_CUDA_TRY(cudaMemsetAsync(state_mem, 0, 16 + 8 * (size_t)tiles, c.stream));
    k_scan_u32<<<(unsigned)tiles, SCAN_THREADS, 0, c.stream>>>(
        in, flags, out, n, (uint32_t *)state_mem, (unsigned long long *)state_mem + 2, total_dev, c.err);
    c.launches++;
    return cudaGetLastError();
}

cudaError_t scan_u32(Ctx &c, const uint32_t *in, const uint8_t *flags, uint32_t *out,
                     int64_t n, uint32_t *total_dev) {
    void *state = nullptr;
    Temps tmp(c);
    if (n > 0) GJ_CUDA_TRY(tmp.alloc_bytes(&state, scan_u32_state_bytes(n)));
    return scan_u32_in(c, in, flags, out, n, total_dev, state, scan_u32_state_bytes(n));
}

cudaError_t scan_u64_sat(Ctx &c, const uint64_t *in, uint64_t *out, int64_t n, uint64_t *total_dev) {
    if (n <= 0) {
        if (total_dev) GJ_CUDA_TRY(cudaMemsetAsync(total_dev, 0, sizeof(uint64_t), c.stream));
        return cudaSuccess;
    }
    const int64_t tiles = ceil_div(n, U64_TILE);
    if (tiles > 0x7fffffff || ((uintptr_t)in | (uintptr_t)out) & 15) return cudaErrorInvalidValue;
    ulonglong2 *state = nullptr;
    Temps tmp(c);
    GJ_CUDA_TRY(tmp.alloc(&state, tiles + 1));
    GJ_CUDA_TRY(cudaMemsetAsync(state, 0, sizeof(ulonglong2) * (size_t)(tiles + 1), c.stream));
    k_scan_u64_sat<<<(unsigned)tiles, U64_THREADS, 0, c.stream>>>((const ulonglong2 *)in, (ulonglong2 *)out, n,
                                                                  (uint32_t *)state, state + 1, total_dev, c.err);
    c.launches++;
    return cudaGetLastError();
}

}  // namespace gj

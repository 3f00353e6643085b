// Exclusive prefix sums that turn per-row and per-slot counts into offsets.
// One launch of one CTA up to kOneCta elements (a solve's scans mostly are
// that short, and a launch costs 2.5 to 4 us on either side); above that two:
// per-tile sums, then the per-tile scan, whose CTAs add up the sums of the
// tiles before theirs themselves.  out[n] receives the total.  Deterministic
// (integer addition).
#include "rdm_internal.cuh"

namespace rdm {
namespace {

constexpr int kThreads = 512;
constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;
constexpr int kOneCta = 4 * kTile;

template <class T>
__device__ T block_exclusive_scan(T v, T *sh, T *total) {
    // warp-shuffle scan then scan of the warp totals
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    if (wid == 0) {
        T w = (lane < (kThreads / 32)) ? sh[lane] : T(0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < (kThreads / 32)) sh[lane] = w;
    }
    __syncthreads();
    T excl = x - v + (wid > 0 ? sh[wid - 1] : T(0));
    if (total) *total = sh[kThreads / 32 - 1];
    __syncthreads();
    return excl;
}

// where the prefix sums go: one array, or the two halves of packed counts
template <class T>
struct Plain {
    T *out;
    __device__ void put(int64_t i, T v) const { out[i] = v; }
};
struct Halves {
    int *lo, *hi;
    __device__ void put(int64_t i, int64_t v) const {
        lo[i] = (int)(v & 0xffffffffll);
        hi[i] = (int)(v >> 32);
    }
};

// the tile of kTile elements at `base`, with `carry` added; returns its total
template <class In, class T, class Dst>
__device__ T scan_tile(const In *in, int64_t base0, int n, T carry, const Dst &dst, T *sh) {
    const int64_t base = base0 + (int64_t)threadIdx.x * kItems;
    T v[kItems], s = 0;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        v[k] = base + k < n ? (T)in[base + k] : T(0);
        s += v[k];
    }
    T tot;
    T e = block_exclusive_scan<T>(s, sh, &tot) + carry;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        if (base + k < n) dst.put(base + k, e);
        e += v[k];
    }
    return tot;
}

template <class In, class T, class Dst>
__global__ void __launch_bounds__(kThreads) k_scan_one(const In *in, int n, Dst dst) {
    __shared__ T sh[32];
    T carry = 0;
    for (int64_t base = 0; base < n; base += kTile) carry += scan_tile<In, T, Dst>(in, base, n, carry, dst, sh);
    if (threadIdx.x == 0) dst.put(n, carry);
}

template <class In, class T>
__global__ void __launch_bounds__(kThreads) k_tile_sums(const In *__restrict__ in, int n, T *__restrict__ tile_sum) {
    __shared__ T sh[32];
    const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kItems;
    T s = 0;
#pragma unroll
    for (int k = 0; k < kItems; ++k)
        if (base + k < n) s += (T)in[base + k];
    T tot;
    block_exclusive_scan<T>(s, sh, &tot);
    if (threadIdx.x == 0) tile_sum[blockIdx.x] = tot;
}

template <class In, class T, class Dst>
__global__ void __launch_bounds__(kThreads) k_scan_apply(const In *in, int n,
                                                         const T *__restrict__ tile_sum, Dst dst) {
    __shared__ T sh[32];
    // sum of the tiles before this one
    T s = 0, before;
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += kThreads) s += tile_sum[k];
    block_exclusive_scan<T>(s, sh, &before);
    const T tot = scan_tile<In, T, Dst>(in, (int64_t)blockIdx.x * kTile, n, before, dst, sh);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) dst.put(n, before + tot);
}

template <class In, class T, class Dst>
void scan_impl(const In *in, Dst dst, int n, T *tmp, cudaStream_t st) {
    if (n <= kOneCta) {
        k_scan_one<In, T, Dst><<<1, kThreads, 0, st>>>(in, n, dst);
        RDM_LAUNCH_CHECK();
        return;
    }
    const int ntiles = (n + kTile - 1) / kTile;
    k_tile_sums<In, T><<<ntiles, kThreads, 0, st>>>(in, n, tmp);
    RDM_LAUNCH_CHECK();
    k_scan_apply<In, T, Dst><<<ntiles, kThreads, 0, st>>>(in, n, tmp, dst);
    RDM_LAUNCH_CHECK();
}

}  // namespace

size_t scan_tmp_elems(int n) { return (size_t)((n + kTile - 1) / kTile + 1); }

void scan_exclusive_i64(const int *in, int64_t *out, int n, int64_t *tmp, cudaStream_t st) {
    scan_impl<int, int64_t>(in, Plain<int64_t>{out}, n, tmp, st);
}
void scan_exclusive_pair(const int64_t *in, int *out_lo, int *out_hi, int n, int64_t *tmp, cudaStream_t st) {
    scan_impl<int64_t, int64_t>(in, Halves{out_lo, out_hi}, n, tmp, st);
}

}  // namespace rdm

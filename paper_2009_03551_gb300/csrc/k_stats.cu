// Reductions in FP64: the trace test of Eq. TC2, the idempotency error, the
// band energies of the stopping rule (Sec. 2.2: E0 = Tr(P0 H0),
// E1 = Tr(P1 H0)), and the polarizability trace (Eq. polar).
//
// Every reduction is two-stage and deterministic: one CTA (or `parts` of them)
// per block row writes partial sums (warp-shuffle reductions, added in a fixed
// order), then one CTA per (system, quantity) adds the rows in a fixed order.
// The branch decision therefore never depends on atomic ordering.
#include <algorithm>

#include "rdm_internal.cuh"

namespace rdm {
namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Column j of a sorted row, or -1: the warp compares 32 columns at a time, two
// independent loads for a row of up to 64 blocks where a binary search would
// wait for six dependent ones.
__device__ __forceinline__ int warp_find_col(const int *__restrict__ col, int lo, int hi, int j, int lane) {
    for (int base = lo; base < hi; base += 64) {
        const int p = base + lane, q = p + 32;
        const int c0 = p < hi ? col[p] : -1, c1 = q < hi ? col[q] : -1;
        const unsigned m0 = __ballot_sync(0xffffffffu, c0 == j), m1 = __ballot_sync(0xffffffffu, c1 == j);
        if (m0) return base + __ffs(m0) - 1;
        if (m1) return base + 31 + __ffs(m1);
    }
    return -1;
}

// row_part layout: [q][NB * parts], q = 0 trace, 1 sumsq, 2 E0, 3+m-1 E1 of
// matrix m.  A block row is shared by `parts` CTAs (consecutive entries), warps
// over blocks, lanes over elements; the warp partials are added in a fixed
// order.  Tr X0 and ||X0||_F^2 run over the blocks of X0, the band energies
// Tr(X H0) only over the blocks of H0 (where H0 is zero they get no
// contribution), each looking up the matching block of X.  The matrices are
// symmetric: only blocks on and above the diagonal are read, those above
// count twice.  Bound by the FP64 pipe (2 FMAs per clock and SM), hence the
// upper triangle only and `parts` for systems with fewer block rows than would
// fill the chip (38 block rows, 1,300 blocks of X0: 155 -> 43 us; 1,250 block
// rows, 110,000 blocks: 0.9 -> 0.5 ms).
constexpr int kStatWarps = 8;
constexpr int kStatQ = 3 + 7;    // up to 7 first-order matrices

__global__ void __launch_bounds__(kStatWarps * 32) k_row_stats(
    const int *__restrict__ rp, const int *__restrict__ col, const double *__restrict__ val, int nmat, int NB, int b,
    const int *__restrict__ hrp, const int *__restrict__ hcol, const double *__restrict__ hval, int parts,
    double *__restrict__ row_part) {
    __shared__ double sh[kStatWarps][kStatQ];
    const int i = blockIdx.x / parts, part = blockIdx.x % parts;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int first = part * kStatWarps + wid, stride = parts * kStatWarps;
    const int bb = b * b;
    double q[kStatQ];
#pragma unroll
    for (int k = 0; k < kStatQ; ++k) q[k] = 0.0;
    // trace and squared norm of X0 (first: the warp's first block of the row)
    for (int p = rp[i] + first; p < rp[i + 1]; p += stride) {
        const int j = col[p];
        if (j < i) continue;
        const double *x = val + (size_t)p * bb;
        double s0 = 0.0, s1 = 0.0;
        int e = lane;
        for (; e + 96 < bb; e += 128) {
            const double v0 = x[e], v1 = x[e + 32], v2 = x[e + 64], v3 = x[e + 96];
            s0 = fma(v0, v0, s0);
            s1 = fma(v1, v1, s1);
            s0 = fma(v2, v2, s0);
            s1 = fma(v3, v3, s1);
        }
        for (; e < bb; e += 32) s0 = fma(x[e], x[e], s0);
        q[1] += j == i ? s0 + s1 : 2.0 * (s0 + s1);
        if (j == i)
            for (int r = lane; r < b; r += 32) q[0] += x[(size_t)r * (b + 1)];
    }
    // band energies over the pattern of H0
    for (int ph = hrp[i] + first; ph < hrp[i + 1]; ph += stride) {
        const int j = hcol[ph];
        if (j < i) continue;
        const double *h = hval + (size_t)ph * bb;
        for (int m = 0; m < nmat; ++m) {
            const int *rpm = rp + (size_t)m * NB;
            const int p = warp_find_col(col, rpm[i], rpm[i + 1], j, lane);
            if (p < 0) continue;
            const double *x = val + (size_t)p * bb;
            double e0 = 0.0, e1 = 0.0;
            int e = lane;
            for (; e + 96 < bb; e += 128) {
                const double v0 = x[e], v1 = x[e + 32], v2 = x[e + 64], v3 = x[e + 96];
                const double h0 = h[e], h1 = h[e + 32], h2 = h[e + 64], h3 = h[e + 96];
                e0 = fma(v0, h0, e0);
                e1 = fma(v1, h1, e1);
                e0 = fma(v2, h2, e0);
                e1 = fma(v3, h3, e1);
            }
            for (; e < bb; e += 32) e0 = fma(x[e], h[e], e0);
            const double eb = j == i ? e0 + e1 : 2.0 * (e0 + e1);
#pragma unroll
            for (int k = 0; k < kStatQ - 2; ++k)
                if (k == m) q[2 + k] += eb;
        }
    }
#pragma unroll
    for (int k = 0; k < kStatQ; ++k) {
        if (k >= 2 + nmat) break;
        const double v = warp_sum(q[k]);
        if (lane == 0) sh[wid][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < 2 + nmat) {
        const int k = threadIdx.x;
        double t = 0.0;
        for (int w = 0; w < kStatWarps; ++w) t += sh[w][k];
        row_part[(size_t)k * NB * parts + blockIdx.x] = t;
    }
}

// Tr X and ||X||_F^2 of one matrix over all its blocks, row_part layout [2][NB]
// (the Newton-Schulz iteration stops on ||X||^2 - 2 Tr X + n, a difference at
// the rounding level, so its sums keep one order)
__global__ void __launch_bounds__(kStatWarps * 32) k_row_trace_norm(const int *__restrict__ rp, const int *__restrict__ col,
                                                                     const double *__restrict__ val, int NB, int b,
                                                                     double *__restrict__ row_part) {
    __shared__ double sh[kStatWarps][2];
    const int i = blockIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int bb = b * b;
    double tr = 0.0, ss = 0.0;
    for (int p = rp[i] + wid; p < rp[i + 1]; p += kStatWarps) {
        const double *x = val + (size_t)p * bb;
        const bool dg = col[p] == i;
        for (int e = lane; e < bb; e += 32) {
            const double v = x[e];
            ss = fma(v, v, ss);
            if (dg && (e / b) == (e % b)) tr += v;
        }
    }
    tr = warp_sum(tr);
    ss = warp_sum(ss);
    if (lane == 0) {
        sh[wid][0] = tr;
        sh[wid][1] = ss;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double t = 0.0;
        for (int w = 0; w < kStatWarps; ++w) t += sh[w][threadIdx.x];
        row_part[(size_t)threadIdx.x * NB + i] = t;
    }
}

// <P_d, H_g> summed over the blocks present in both, per row:
// row_part[(g*np + d)][NB]; one CTA per block row and (g, d), warps over the
// blocks of H_g
__global__ void __launch_bounds__(128) k_row_dots(const int *__restrict__ prp, const int *__restrict__ pcol,
                                                  const double *__restrict__ pval, int np,
                                                  const int *__restrict__ hrp, const int *__restrict__ hcol,
                                                  const double *__restrict__ hval, int nh, int NB, int b,
                                                  double *__restrict__ row_part) {
    __shared__ double sh[4];
    const int i = blockIdx.x, g = blockIdx.y / np, d = blockIdx.y % np;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int bb = b * b;
    const int *hr = hrp + (size_t)g * NB, *pr = prp + (size_t)d * NB;
    double acc = 0.0;
    for (int q = hr[i] + wid; q < hr[i + 1]; q += 4) {
        const int p = warp_find_col(pcol, pr[i], pr[i + 1], hcol[q], lane);
        if (p < 0) continue;
        const double *x = pval + (size_t)p * bb;
        const double *h = hval + (size_t)q * bb;
#pragma unroll 4
        for (int e = lane; e < bb; e += 32) acc = fma(x[e], h[e], acc);
    }
    acc = warp_sum(acc);
    if (lane == 0) sh[wid] = acc;
    __syncthreads();
    if (threadIdx.x == 0) row_part[(size_t)blockIdx.y * NB + i] = (sh[0] + sh[1]) + (sh[2] + sh[3]);
}

// out[s*nq + q] = sum_{i in system s} row_part[q][i], fixed order
__global__ void k_sys_sum(const double *__restrict__ row_part, int nq, int NB,
                          const int *__restrict__ row0, const int *__restrict__ nbs, int parts,
                          double *__restrict__ out) {
    __shared__ double sh[32];
    int s = blockIdx.x, q = blockIdx.y;
    const double *r = row_part + ((size_t)q * NB + row0[s]) * parts;
    double acc = 0.0;
    for (int i = threadIdx.x; i < nbs[s] * parts; i += blockDim.x) acc += r[i];
    acc = warp_sum(acc);
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) sh[w] = acc;
    __syncthreads();
    if (w == 0) {
        double v = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
        v = warp_sum(v);
        if (lane == 0) out[(size_t)s * nq + q] = v;
    }
}

}  // namespace

int row_stats_parts(int NB) {
    // enough CTAs for four per SM, at most one per warp's worth of a row of 64 blocks
    return std::max(1, std::min(8, 608 / std::max(NB, 1)));
}

void launch_row_stats(const int *row_ptr, const int *col, const double *val, int nmat, int NB,
                      int b, const int *h_row_ptr, const int *h_col, const double *h_val, int parts,
                      double *row_part, cudaStream_t st) {
    if (NB == 0) return;
    if (nmat > kStatQ - 2) throw Error{-1, "at most 7 first-order matrices"};
    k_row_stats<<<(unsigned)NB * parts, kStatWarps * 32, 0, st>>>(row_ptr, col, val, nmat, NB, b, h_row_ptr, h_col,
                                                                  h_val, parts, row_part);
    RDM_LAUNCH_CHECK();
}

void launch_row_trace_norm(const int *row_ptr, const int *col, const double *val, int NB, int b, double *row_part,
                           cudaStream_t st) {
    if (NB == 0) return;
    k_row_trace_norm<<<NB, kStatWarps * 32, 0, st>>>(row_ptr, col, val, NB, b, row_part);
    RDM_LAUNCH_CHECK();
}

void launch_row_dots(const int *p_row_ptr, const int *p_col, const double *p_val, int np,
                     const int *h_row_ptr, const int *h_col, const double *h_val, int nh,
                     int NB, int b, double *row_part, cudaStream_t st) {
    if (NB == 0 || np == 0 || nh == 0) return;
    k_row_dots<<<dim3(NB, np * nh), 128, 0, st>>>(p_row_ptr, p_col, p_val, np, h_row_ptr, h_col, h_val, nh, NB, b,
                                                  row_part);
    RDM_LAUNCH_CHECK();
}

void launch_sys_sum(const double *row_part, int nq, int NB, const int *row0, const int *nbs,
                    int S, double *out, cudaStream_t st, int parts) {
    if (S == 0 || nq == 0) return;
    k_sys_sum<<<dim3(S, nq), 256, 0, st>>>(row_part, nq, NB, row0, nbs, parts, out);
    RDM_LAUNCH_CHECK();
}

}  // namespace rdm

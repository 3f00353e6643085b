// Reductions in FP64: the trace test of Eq. TC2, the idempotency error, the
// band energies of the stopping rule (Sec. 2.2: E0 = Tr(P0 H0),
// E1 = Tr(P1 H0)), and the polarizability trace (Eq. polar).
//
// Every reduction is two-stage and deterministic: warps write partial sums of
// their block row (warp-shuffle reductions), then one CTA per (system,
// quantity) adds them, row by row, in a fixed order.
// The branch decision therefore never depends on atomic ordering.
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

// row_part layout: [q][NB][kStatWarps], q = 0 trace, 1 sumsq, 2 E0, 3+m-1 E1 of
// matrix m.  Warp w of block row i adds the blocks w, w + 8, ... of the row,
// lanes over elements; Tr X0 and ||X0||_F^2 run over the blocks of X0, the band
// energies Tr(X H0) only over the blocks of H0 (where H0 is zero they get no
// contribution), each looking up the matching block of X.  k_sys_sum adds the
// warps' sums of a row in order.  A sum that ends within its rounding of an
// integer decides a branch (Tr X0 against N_occ at convergence), so the order
// of the additions is fixed: per warp and lane one chain over the blocks and
// elements of its share.  Bound by the FP64 pipe (2 FMAs per clock and SM); the
// chains of a row (8 warps, 2 + nmat sums) are spread over 2 (1 + nmat) CTAs, so
// that a system of few block rows fills the chip (38 block rows, 1,300 blocks of
// X0: 155 us in one CTA per row, 27 us spread, 22 us with the next 256
// elements of a warp's share loaded while these are added, and with the blocks
// of X looked up by 32 lanes at once).
constexpr int kStatWarps = 8;    // warps per block row
constexpr int kStatCta = 4;      // of them in one CTA

// 256 elements, a lane every 32nd
__device__ __forceinline__ void load8(double (&v)[8], const double *__restrict__ x) {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = x[32 * k];
}

__global__ void __launch_bounds__(kStatCta * 32) k_row_stats(
    const int *__restrict__ rp, const int *__restrict__ col, const double *__restrict__ val, int NB, int b,
    const int *__restrict__ hrp, const int *__restrict__ hcol, const double *__restrict__ hval,
    double *__restrict__ row_part) {
    const int lane = threadIdx.x & 31;
    const int slot = blockIdx.x * kStatCta + (threadIdx.x >> 5);     // row, warp of the row
    const int i = slot / kStatWarps, w = slot % kStatWarps;
    const int bb = b * b, n8 = bb >> 8;          // 256 elements at a time (blocks of 16 and more)
    const size_t nslot = (size_t)NB * kStatWarps;
    if (blockIdx.y == 0) {
        // trace and squared norm of X0
        double tr = 0.0, ss = 0.0;
        int p = rp[i] + w;
        const int end = rp[i + 1];
        double v[8], nx[8];
        if (n8 && p < end) load8(v, val + (size_t)p * bb + lane);
        for (; p < end; p += kStatWarps) {
            const double *x = val + (size_t)p * bb;
            for (int q = 0; q < n8; ++q) {
                const int pn = q + 1 < n8 ? p : p + kStatWarps;
                if (pn < end) load8(nx, val + (size_t)pn * bb + (q + 1 < n8 ? 256 * (q + 1) : 0) + lane);
#pragma unroll
                for (int k = 0; k < 8; ++k) ss = fma(v[k], v[k], ss);
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = nx[k];
            }
            for (int e = 256 * n8 + lane; e < bb; e += 32) ss = fma(x[e], x[e], ss);
            if (col[p] == i)
                // the lane's elements in order, those on the diagonal
                for (int e = 0; e < bb; e += b + 1)
                    if ((e & 31) == lane) tr += x[e];
        }
        tr = warp_sum(tr);
        ss = warp_sum(ss);
        if (lane == 0) {
            row_part[slot] = tr;
            row_part[nslot + slot] = ss;
        }
        return;
    }
    // band energy of matrix m over the pattern of H0
    const int m = blockIdx.y - 1;
    const int *rpm = rp + (size_t)m * NB;
    const int lo = rpm[i], hi = rpm[i + 1], hend = hrp[i + 1];
    double q = 0.0;
    for (int first = hrp[i] + w; first < hend; first += 32 * kStatWarps) {
        const int ph = first + kStatWarps * lane;
        int mine = -1;                           // the block of X at H0's block ph
        if (ph < hend) {
            const int j = hcol[ph];
            int a = lo, z = hi;
            while (a < z) {
                const int mid = (a + z) >> 1;
                if (col[mid] < j) a = mid + 1; else z = mid;
            }
            if (a < hi && col[a] == j) mine = a;
        }
        unsigned todo = __ballot_sync(0xffffffffu, mine >= 0);
        if (!todo) continue;
        int u = __ffs(todo) - 1;
        const double *x = val + (size_t)__shfl_sync(0xffffffffu, mine, u) * bb + lane;
        const double *h = hval + (size_t)(first + kStatWarps * u) * bb + lane;
        double v[8], g[8], nv[8], ng[8];
        if (n8) {
            load8(v, x);
            load8(g, h);
        }
        for (;;) {
            todo &= todo - 1;
            u = todo ? __ffs(todo) - 1 : 0;
            const double *xn = val + (size_t)__shfl_sync(0xffffffffu, mine, u) * bb + lane;
            const double *hn = hval + (size_t)(first + kStatWarps * u) * bb + lane;
            double eb = 0.0;
            for (int k8 = 0; k8 < n8; ++k8) {
                if (k8 + 1 < n8) {
                    load8(nv, x + 256 * (k8 + 1));
                    load8(ng, h + 256 * (k8 + 1));
                } else if (todo) {
                    load8(nv, xn);
                    load8(ng, hn);
                }
#pragma unroll
                for (int k = 0; k < 8; ++k) eb = fma(v[k], g[k], eb);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    v[k] = nv[k];
                    g[k] = ng[k];
                }
            }
            for (int e = 256 * n8; e + lane < bb; e += 32) eb = fma(x[e], h[e], eb);
            q += eb;
            if (!todo) break;
            x = xn;
            h = hn;
        }
    }
    q = warp_sum(q);
    if (lane == 0) row_part[(2 + m) * nslot + slot] = q;
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
    for (int i = threadIdx.x; i < nbs[s]; i += blockDim.x) {
        double t = parts > 1 ? 0.0 : r[i];
        if (parts > 1)
            for (int w = 0; w < parts; ++w) t += r[(size_t)i * parts + w];
        acc += t;
    }
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

int row_stats_parts() { return kStatWarps; }

void launch_row_stats(const int *row_ptr, const int *col, const double *val, int nmat, int NB,
                      int b, const int *h_row_ptr, const int *h_col, const double *h_val,
                      double *row_part, cudaStream_t st) {
    if (NB == 0) return;
    k_row_stats<<<dim3((unsigned)NB * (kStatWarps / kStatCta), 1 + nmat), kStatCta * 32, 0, st>>>(
        row_ptr, col, val, NB, b, h_row_ptr, h_col, h_val, row_part);
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

// Numeric phase on the CUDA cores (FP64 and FP32 operands), with the update
// and truncation of Eqs. TC2 / TC2-CPSCF fused into the epilogue:
//
//   C_ij = c_lin X_ij + c_sq sum_{(a,b) in pairs(i,j)} A_a (B_b)^T
//
// for every upper-triangle output block (j >= i); the lower block (j,i) is
// written as the transpose, so the result is exactly symmetric.  Diagonal
// blocks are symmetrised ((C + C^T)/2) because the accumulation order of
// C_mn and C_nm differs.  The block Frobenius norm is reduced in FP64 and the
// block is kept iff norm >= tau (the block-wise "filter" of Sec. 2.3).
//
// One CTA per output block (work items from an atomic counter) for b >= 8; the
// two operand blocks of each pair are staged in shared memory, each thread owns
// ceil(b^2 / threads) outputs.  On GB300 the FP64 rate is the bound of this
// kernel; the FP32 variant converts the FP64 master values on load.
#include "fp_bits.cuh"
#include "rdm_internal.cuh"

#include <algorithm>
#include <type_traits>

namespace rdm {
namespace {

template <int B>
struct Cfg {
    static constexpr int NT = B * B >= 256 ? 256 : B * B;      // B = 8 and up
    static constexpr int PER = (B * B + NT - 1) / NT;
    static constexpr int LD = B + 1;
};

__device__ __forceinline__ double block_sum(double v, double *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double t = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += sh[k];
    __syncthreads();
    return t;
}

template <class T>
__device__ __forceinline__ T operand(double x) {
    if constexpr (std::is_same<T, float>::value) return f64_to_f32(x);
    else return x;
}

// B consecutive doubles (a row of a block, aligned to its size)
template <int B>
__device__ __forceinline__ void load_row(const double *p, double (&v)[B]) {
    if constexpr (B == 4) {
        ld_f64x4(p, v);
    } else if constexpr (B == 2) {
        const double2 x = *reinterpret_cast<const double2 *>(p);
        v[0] = x.x;
        v[1] = x.y;
    } else {
        v[0] = p[0];
    }
}

template <int B, class T>
__global__ void __launch_bounds__(Cfg<B>::NT) k_numeric_simt(NumArgs a) {
    constexpr int NT = Cfg<B>::NT, PER = Cfg<B>::PER, LD = Cfg<B>::LD, BB = B * B;
    extern __shared__ double smem_d[];
    T *As = reinterpret_cast<T *>(smem_d);
    T *Bs = As + B * LD;
    double *Cs = smem_d;                    // reused for the epilogue (B*LD doubles)
    __shared__ double red[32];
    const int tid = threadIdx.x;

    __shared__ int s_w;
    const int nwork = *a.nwork;
    for (;;) {
        // work items are handed out in list order by an atomic counter, so the
        // blocks in flight stay close in the list and share operands in L2
        if (threadIdx.x == 0) s_w = atomicAdd(a.work_next, 1);
        __syncthreads();
        const int w = s_w;
        __syncthreads();
        if (w >= nwork) break;
        const int s = a.work[w];
        const int i = a.slot_row[s];
        const int sys = a.sys_of_row[i];
        const int job = a.slot_job[s];
        const double cl = a.c_lin[sys], cq = a.c_sq[sys];
        const double tau = a.job_tau_sel[job] ? a.tau1[sys] : a.tau0[sys];
        const int64_t p0 = a.pair_off ? a.pair_off[s] : 0, p1 = a.pair_off ? a.pair_off[s + 1] : 0;
        const int st = a.slot_t[s], sx = a.slot_x[s];

        T acc[PER];
#pragma unroll
        for (int r = 0; r < PER; ++r) acc[r] = T(0);

        for (int64_t q = p0; q < p1; ++q) {
            const double *ga = a.in_val + (size_t)a.pair_a[q] * BB;
            const double *gb = a.in_val + (size_t)a.pair_b[q] * BB;
            __syncthreads();
            for (int e = tid; e < BB; e += NT) {
                As[(e / B) * LD + (e % B)] = operand<T>(ga[e]);
                Bs[(e / B) * LD + (e % B)] = operand<T>(gb[e]);
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int e = tid + r * NT;
                if (e < BB) {
                    const int m = e / B, n = e % B;
                    const T *ar = As + m * LD;
                    const T *br = Bs + n * LD;
                    T sacc = acc[r];
#pragma unroll 8
                    for (int kk = 0; kk < B; ++kk) sacc = fma(ar[kk], br[kk], sacc);
                    acc[r] = sacc;
                }
            }
        }

        // epilogue: linear term, symmetrisation, norm, truncation (the lower
        // triangle is written by the compaction, as the transpose)
        double out[PER];
        const double *gx = sx >= 0 ? a.in_val + (size_t)sx * BB : nullptr;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            const int e = tid + r * NT;
            if (e < BB) {
                double v = cq * (double)acc[r];
                if (gx) v = fma(cl, gx[e], v);
                out[r] = v;
                Cs[(e / B) * LD + (e % B)] = v;
            }
        }
        __syncthreads();
        const bool diag = (st == s);
        double ss = 0.0;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            const int e = tid + r * NT;
            if (e < BB) {
                if (diag) {
                    const int m = e / B, n = e % B;
                    out[r] = 0.5 * (Cs[m * LD + n] + Cs[n * LD + m]);
                }
                ss += out[r] * out[r];
            }
        }
        const double nrm = sqrt(block_sum(ss, red));
        const bool keep = (nrm >= tau) && (nrm > 0.0);
        double *o = a.out_val + (size_t)(a.uidx[s] - a.u0) * BB;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            const int e = tid + r * NT;
            if (e < BB) o[e] = out[r];
        }
        if (tid == 0) {
            a.out_nrm[s] = __double2float_ru(nrm);
            a.keep[s] = keep;
        }
    }
}

// ---------------------------------------------------------------------------
// Blocks of 1, 2 and 4: b*b lanes per output block, a lane its element, rows of
// the operand blocks read straight into registers, four pairs ahead of the
// FMAs.  With so few operations per pair the kernel waits for loads; staging
// each pair in shared memory between barriers, with half of a CTA's 32 threads
// idle at b = 4, took 87 us for the 4,160 blocks of up to 128 pairs of a
// 64-atom chain, 59 us here, 5 more than its FMAs take on the FP64 pipe.  Same chains of FMAs and the same sums as
// k_numeric_simt.
// ---------------------------------------------------------------------------
template <int B, class T>
__global__ void __launch_bounds__(128) k_numeric_small(NumArgs a) {
    constexpr int L = B * B, PB = 128 / L, BB = B * B, U = 4;
    __shared__ int s_w;
    const int nwork = *a.nwork;
    const int g = threadIdx.x / L, e = threadIdx.x % L, m = e / B, n = e % B;
    for (;;) {
        if (threadIdx.x == 0) s_w = atomicAdd(a.work_next, PB);
        __syncthreads();
        const int w0 = s_w, w = w0 + g;
        __syncthreads();
        if (w0 >= nwork) break;
        const bool on = w < nwork;
        const int s = on ? a.work[w] : 0;
        const int64_t p0 = on && a.pair_off ? a.pair_off[s] : 0, p1 = on && a.pair_off ? a.pair_off[s + 1] : 0;
        T acc = T(0);
        int64_t q = p0;
        for (; q + U <= p1; q += U) {
            double x[U][B], y[U][B];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                load_row<B>(a.in_val + (size_t)a.pair_a[q + u] * BB + m * B, x[u]);
                load_row<B>(a.in_val + (size_t)a.pair_b[q + u] * BB + n * B, y[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int k = 0; k < B; ++k) acc = fma(operand<T>(x[u][k]), operand<T>(y[u][k]), acc);
        }
        for (; q < p1; ++q) {
            double x[B], y[B];
            load_row<B>(a.in_val + (size_t)a.pair_a[q] * BB + m * B, x);
            load_row<B>(a.in_val + (size_t)a.pair_b[q] * BB + n * B, y);
#pragma unroll
            for (int k = 0; k < B; ++k) acc = fma(operand<T>(x[k]), operand<T>(y[k]), acc);
        }
        double out = 0.0, tau = 0.0;
        bool diag = false;
        if (on) {
            const int sys = a.sys_of_row[a.slot_row[s]];
            const int job = a.slot_job[s], sx = a.slot_x[s];
            tau = a.job_tau_sel[job] ? a.tau1[sys] : a.tau0[sys];
            out = a.c_sq[sys] * (double)acc;
            if (sx >= 0) out = fma(a.c_lin[sys], a.in_val[(size_t)sx * BB + e], out);
            diag = a.slot_t[s] == s;
        }
        const double tr = __shfl_sync(0xffffffffu, out, (threadIdx.x & 31) - e + n * B + m);
        if (diag) out = 0.5 * (out + tr);
        double ss = out * out;
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        if (on) {
            const double nrm = sqrt(ss);
            a.out_val[(size_t)(a.uidx[s] - a.u0) * BB + e] = out;
            if (e == 0) {
                a.out_nrm[s] = __double2float_ru(nrm);
                a.keep[s] = (nrm >= tau) && (nrm > 0.0);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Double-FP32 products of 32 x 32 blocks: 64 threads per output block, each a
// 4 x 4 register tile at rows r0 + 8i and columns c0 + 8j (r0 = t/8,
// c0 = t%8), so that the 16-byte shared-memory reads of a quarter warp hit 8
// different banks (B rows) or broadcast (A rows).  Operand blocks come from
// the FP32 (hi, lo) copies of the master values, double-buffered with
// cp.async.
// ---------------------------------------------------------------------------
constexpr int kF32Ld = 36;   // padded row stride in floats (144 B, 16-byte aligned)

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Double-FP32 ("float-float") products of the FP64 masters split as
// x = hi + lo (two FP32 planes): the
// hi*hi products are accumulated without rounding loss by the error-free
// transformations of Ogita, Rump and Oishi (2005) -- the exact product
// p + e = hi_a hi_b from one multiply and one fused multiply-add, the exact
// sum s + t = acc + p from six additions -- and the small cross terms hi*lo
// and lo*hi are added in plain FP32 into the low word.  The result carries
// about 46 bits, enough for FP64-class refinement of X0^2, on the FP32 pipe.
__global__ void __launch_bounds__(64) k_numeric_ff_b32(NumArgs a) {
    constexpr int NP = 2;                          // operand planes (hi, lo)
    __shared__ __align__(16) float sA[2][NP][32 * kF32Ld];
    __shared__ __align__(16) float sB[2][NP][32 * kF32Ld];
    __shared__ double sC[32 * 33];
    __shared__ float red[2];
    const int tid = threadIdx.x;
    const int r0 = tid >> 3, c0 = tid & 7;
    const float *planes[2] = {a.in_f32, a.in_f32lo};

    __shared__ int s_w;
    const int nwork = *a.nwork;
    for (;;) {
        // work items are handed out in list order by an atomic counter, so the
        // blocks in flight stay close in the list and share operands in L2
        if (threadIdx.x == 0) s_w = atomicAdd(a.work_next, 1);
        __syncthreads();
        const int w = s_w;
        __syncthreads();
        if (w >= nwork) break;
        const int s = a.work[w];
        const int i = a.slot_row[s];
        const int sys = a.sys_of_row[i];
        const int job = a.slot_job[s];
        const double tau = a.job_tau_sel[job] ? a.tau1[sys] : a.tau0[sys];
        const int64_t p0 = a.pair_off ? a.pair_off[s] : 0, p1 = a.pair_off ? a.pair_off[s + 1] : 0;
        const int st = a.slot_t[s], sx = a.slot_x[s];

        float acc[4][4], accl[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = accl[u][v] = 0.f;

        auto issue = [&](int64_t q, int buf) {
#pragma unroll
            for (int pl = 0; pl < NP; ++pl) {
                const float *ga = planes[pl] + (size_t)a.pair_a[q] * 1024;
                const float *gb = planes[pl] + (size_t)a.pair_b[q] * 1024;
#pragma unroll
                for (int c = tid; c < 256; c += 64) {
                    const int row = c >> 3, col4 = (c & 7) * 4;
                    cp_async16(&sA[buf][pl][row * kF32Ld + col4], ga + row * 32 + col4);
                    cp_async16(&sB[buf][pl][row * kF32Ld + col4], gb + row * 32 + col4);
                }
            }
            cp_async_commit();
        };
        __syncthreads();
        if (p0 < p1) issue(p0, 0);
        for (int64_t q = p0; q < p1; ++q) {
            const int buf = (int)((q - p0) & 1);
            if (q + 1 < p1) {
                issue(q + 1, buf ^ 1);
                cp_async_wait1();
            } else {
                cp_async_wait0();
            }
            __syncthreads();
            const float *A_ = sA[buf][0];
            const float *B_ = sB[buf][0];
            // the double-FP32 body is large: not unrolled over kk, so that the
            // loop stays in the instruction cache
#pragma unroll 1
            for (int kk = 0; kk < 32; kk += 4) {
                float4 av[4], bv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) av[u] = *reinterpret_cast<const float4 *>(&A_[(r0 + 8 * u) * kF32Ld + kk]);
#pragma unroll
                for (int v = 0; v < 4; ++v) bv[v] = *reinterpret_cast<const float4 *>(&B_[(c0 + 8 * v) * kF32Ld + kk]);
                {
                    const float *Al = sA[buf][NP - 1];
                    const float *Bl = sB[buf][NP - 1];
                    float4 al[4], bl[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) al[u] = *reinterpret_cast<const float4 *>(&Al[(r0 + 8 * u) * kF32Ld + kk]);
#pragma unroll
                    for (int v = 0; v < 4; ++v) bl[v] = *reinterpret_cast<const float4 *>(&Bl[(c0 + 8 * v) * kF32Ld + kk]);
                    // k outermost: the 16 accumulator chains of the thread are
                    // independent, so consecutive operations do not wait on each other
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float ah = k == 0 ? av[u].x : k == 1 ? av[u].y : k == 2 ? av[u].z : av[u].w;
                            const float alo = k == 0 ? al[u].x : k == 1 ? al[u].y : k == 2 ? al[u].z : al[u].w;
#pragma unroll
                            for (int v = 0; v < 4; ++v) {
                                const float bh = k == 0 ? bv[v].x : k == 1 ? bv[v].y : k == 2 ? bv[v].z : bv[v].w;
                                const float blo = k == 0 ? bl[v].x : k == 1 ? bl[v].y : k == 2 ? bl[v].z : bl[v].w;
                                const float sh = acc[u][v];
                                const float p = __fmul_rn(ah, bh);
                                const float e = fmaf(ah, bh, -p);                // p + e = ah bh exactly
                                const float sn = __fadd_rn(sh, p);
                                const float z = __fsub_rn(sn, sh);
                                const float t = __fadd_rn(__fsub_rn(sh, __fsub_rn(sn, z)), __fsub_rn(p, z));   // sn + t = sh + p
                                acc[u][v] = sn;
                                float sl = accl[u][v];
                                sl = fmaf(ah, blo, sl);
                                sl = fmaf(alo, bh, sl);
                                accl[u][v] = __fadd_rn(sl, __fadd_rn(t, e));
                            }
                        }
                    }
                }
            }
            __syncthreads();
        }

        // epilogue: C = c_lin X + c_sq acc in FP64, symmetrised on the
        // diagonal, norm, truncation
        const double *gx = sx >= 0 ? a.in_val + (size_t)sx * 1024 : nullptr;
        const bool diag = (st == s);
        const double cl = a.c_lin[sys], cq = a.c_sq[sys];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int r = r0 + 8 * u, c = c0 + 8 * v;
                double x = cq * ((double)acc[u][v] + (double)accl[u][v]);
                if (gx) x = fma(cl, gx[r * 32 + c], x);
                sC[r * 33 + c] = x;
            }
        __syncthreads();
        float ss = 0.f;
        if (diag) {
            double sym[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int r = r0 + 8 * u, c = c0 + 8 * v;
                    sym[u][v] = 0.5 * (sC[r * 33 + c] + sC[c * 33 + r]);
                }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) sC[(r0 + 8 * u) * 33 + c0 + 8 * v] = sym[u][v];
            __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const float x = (float)sC[(r0 + 8 * u) * 33 + c0 + 8 * v];
                ss = fmaf(x, x, ss);
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        if ((tid & 31) == 0) red[tid >> 5] = ss;
        __syncthreads();
        const float nrm = sqrtf(red[0] + red[1]) * (1.0f + 1e-6f);
        const bool keep = ((double)nrm >= tau) && (nrm > 0.f);
        double *o = a.out_val + (size_t)(a.uidx[s] - a.u0) * 1024;
        for (int e = tid; e < 1024; e += 64) o[e] = (double)sC[(e >> 5) * 33 + (e & 31)];
        if (tid == 0) {
            a.out_nrm[s] = nrm;
            a.keep[s] = keep;
        }
    }
}

// ---------------------------------------------------------------------------
// FP32 products of 32 x 32 blocks, one warp per output block, two FMAs per
// instruction (fma.rn.f32x2: both halves are IEEE FMAs).  Half-warp kh covers
// k = 16 kh .. 16 kh + 15 of every pair, lane l of it the 8 x 8 tile of rows
// 8 (l / 4) .. and columns 8 (l % 4) ..; per k it reads 8 elements of each
// operand (4 shared-memory reads of 16 bytes for 64 FMAs, 1 byte per FMA).
// The operands are staged as [k][row] and [k][column], which for a symmetric
// matrix is the block at the transposed position as it is stored, so that
// adjacent rows are register pairs as loaded and only the 8 column elements
// are doubled by moves: 52 issue slots per 64 FMAs, whose pipe takes 64 clocks.
// A version with 64 threads per block, 8 x 4 tiles and 16-byte reads along k
// (1.5 bytes per FMA, where a 16-byte warp read takes 4 shared-memory cycles)
// was bound by those reads: 44.5 TFLOP/s with the FMA pipe at 58%; this one 58.6 TFLOP/s (1,000-atom
// cluster, 125 -> 94.5 ms of products).  The
// k-halves' sums and the norm keep the order of that version.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void fma2(unsigned long long &d, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long dup2(float x) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
    return d;
}

__global__ void __launch_bounds__(32, 13) k_numeric_f32_x2(NumArgs a) {
    __shared__ __align__(16) float sm[2][2][1024];         // [buffer][operand][k][row or column]
    float *sC = &sm[0][0][0];                              // 32 x 33, after the products
    const int lane = threadIdx.x;
    const int kh = lane >> 4, l = lane & 15;
    const int r0 = 8 * (l >> 2), c0 = 8 * (l & 3), k0 = 16 * kh;
    const int nwork = *a.nwork;
    for (;;) {
        int w = 0;
        if (lane == 0) w = atomicAdd(a.work_next, 1);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= nwork) break;
        const int s = a.work[w];
        const int i = a.slot_row[s];
        const int sys = a.sys_of_row[i];
        const int job = a.slot_job[s];
        const double tau = a.job_tau_sel[job] ? a.tau1[sys] : a.tau0[sys];
        const int64_t p0 = a.pair_off ? a.pair_off[s] : 0, p1 = a.pair_off ? a.pair_off[s + 1] : 0;
        const int st = a.slot_t[s], sx = a.slot_x[s];

        unsigned long long acc[4][8];                      // rows 2u, 2u + 1 of the tile, column v
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 8; ++v) acc[u][v] = 0ull;
        int na = 0, nb = 0;                                // positions of the next pair to stage
        auto look = [&](int64_t q) {
            if (q < p1) {
                na = max(a.tpos[a.pair_a[q]], 0);     // (-1, a missing transpose, is reported by the host)
                nb = max(a.tpos[a.pair_b[q]], 0);
            }
        };
        auto issue = [&](int buf) {
            const float *ga = a.in_f32 + (size_t)na * 1024 + 4 * lane;
            const float *gb = a.in_f32 + (size_t)nb * 1024 + 4 * lane;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                cp_async16(&sm[buf][0][128 * c + 4 * lane], ga + 128 * c);
                cp_async16(&sm[buf][1][128 * c + 4 * lane], gb + 128 * c);
            }
            cp_async_commit();
        };
        __syncwarp();
        look(p0);
        if (p0 < p1) issue(0);
        look(p0 + 1);
        for (int64_t q = p0; q < p1; ++q) {
            const int buf = (int)((q - p0) & 1);
            if (q + 1 < p1) {
                issue(buf ^ 1);
                look(q + 2);
                cp_async_wait1();
            } else {
                cp_async_wait0();
            }
            __syncwarp();
            const float *A_ = &sm[buf][0][k0 * 32 + r0], *B_ = &sm[buf][1][k0 * 32 + c0];
#pragma unroll 4
            for (int k = 0; k < 16; ++k) {
                const ulonglong2 x0 = *reinterpret_cast<const ulonglong2 *>(A_ + 32 * k);
                const ulonglong2 x1 = *reinterpret_cast<const ulonglong2 *>(A_ + 32 * k + 4);
                const float4 y0 = *reinterpret_cast<const float4 *>(B_ + 32 * k);
                const float4 y1 = *reinterpret_cast<const float4 *>(B_ + 32 * k + 4);
                const unsigned long long x[4] = {x0.x, x0.y, x1.x, x1.y};
                const float y[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    const unsigned long long yy = dup2(y[v]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) fma2(acc[u][v], x[u], yy);
                }
            }
            __syncwarp();
        }

        // P_0 + P_1 (the half-warps hold the same tiles), then C = c_lin X + c_sq P;
        // half-warp kh finishes columns 4 kh .. 4 kh + 3 of each tile
        const float *gx = sx >= 0 ? a.in_f32 + (size_t)sx * 1024 : nullptr;
        const bool diag = (st == s);
        const float cl = (float)a.c_lin[sys], cq = (float)a.c_sq[sys];
        float t[8][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const unsigned long long o = __shfl_xor_sync(0xffffffffu, acc[u][v], 16);
                const float lo = __uint_as_float((unsigned)acc[u][v]) + __uint_as_float((unsigned)o);
                const float hi = __uint_as_float((unsigned)(acc[u][v] >> 32)) + __uint_as_float((unsigned)(o >> 32));
                if ((v >> 2) == kh) {
                    t[2 * u][v & 3] = lo;
                    t[2 * u + 1][v & 3] = hi;
                }
            }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int c = c0 + 4 * kh;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (gx) x = *reinterpret_cast<const float4 *>(gx + (r0 + r) * 32 + c);
            float *o = sC + (r0 + r) * 33 + c;
            o[0] = gx ? fmaf(cl, x.x, cq * t[r][0]) : cq * t[r][0];
            o[1] = gx ? fmaf(cl, x.y, cq * t[r][1]) : cq * t[r][1];
            o[2] = gx ? fmaf(cl, x.z, cq * t[r][2]) : cq * t[r][2];
            o[3] = gx ? fmaf(cl, x.w, cq * t[r][3]) : cq * t[r][3];
        }
        __syncwarp();
        if (diag) {
            // (X + X^T) / 2 of the elements on and above the diagonal, mirrored
            for (int r = 0; r < 32; ++r) {
                float y = 0.f;
                if (lane >= r) y = 0.5f * (sC[r * 33 + lane] + sC[lane * 33 + r]);
                __syncwarp();
                if (lane >= r) sC[r * 33 + lane] = sC[lane * 33 + r] = y;
                __syncwarp();
            }
        }
        float s0 = 0.f, s1 = 0.f;                          // even and odd rows
#pragma unroll
        for (int r = 0; r < 32; r += 2) {
            const float x = sC[r * 33 + lane], y = sC[(r + 1) * 33 + lane];
            s0 = fmaf(x, x, s0);
            s1 = fmaf(y, y, s1);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        }
        const float nrm = sqrtf(s0 + s1) * (1.0f + 1e-6f);
        const bool keep = ((double)nrm >= tau) && (nrm > 0.f);
        float4 *o = reinterpret_cast<float4 *>(a.out_val + (size_t)(a.uidx[s] - a.u0) * 1024);
#pragma unroll
        for (int c = 0; c < 8; ++c) {                      // layout f32_index: 4 columns of row `lane`
            const float *x = &sC[lane * 33 + 4 * c];
            o[c * 32 + lane] = make_float4(x[0], x[1], x[2], x[3]);
        }
        if (lane == 0) {
            a.out_nrm[s] = nrm;
            a.keep[s] = (keep ? kKeepBlock : 0) | kBlockF32;
        }
        __syncwarp();
    }
}

// Diagonal elements of A A (32 x 32 blocks) as FP64 FMA chains, written over
// those of the slice product in out_val.  The trace of X0^2 decides the branch
// of Eq. TC2, at convergence by its last bits (Tr X0 is then N_occ up to
// rounding), so it keeps the rounding of the chains that the CUDA-core kernel
// computes: block by block along the row, k ascending, the linear term last.
// One warp per block row, a lane per element; it waits for its chain (1,600
// dependent FMAs in a row of 50 blocks, ~40 us beside ~2 ms of products).
__global__ void __launch_bounds__(32) k_diag_fp64(const int *__restrict__ rp, const int *__restrict__ out_rp,
                                                  const int *__restrict__ out_col, NumArgs a, JobTable jt, JobMask jobs,
                                                  const int *__restrict__ sys_tier, int NB, int r0, int nrows) {
    const int r = r0 + blockIdx.x, p = r / NB, i = r - p * NB;
    const int lane = threadIdx.x;
    const int sys = a.sys_of_row[i];
    const Job &job = jt.job[p];
    if (!a.active[sys] || job.nterm != 1 || !((jobs.m[sys_tier[sys] & (kMaxTiers - 1)] >> p) & 1u)) return;
    int lo = out_rp[r], hi = out_rp[r + 1];
    const int end = hi;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (out_col[mid] < i) lo = mid + 1; else hi = mid;
    }
    if (lo >= end || out_col[lo] != i) return;             // no diagonal block in the mask
    double acc = 0.0;
    const int q1 = rp[job.a[0] * NB + i + 1];
    for (int q = rp[job.a[0] * NB + i]; q < q1; ++q) {
        const double2 *x = reinterpret_cast<const double2 *>(a.in_val + (size_t)q * 1024 + lane * 32);
        double2 v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = x[k];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            acc = fma(v[k].x, v[k].x, acc);
            acc = fma(v[k].y, v[k].y, acc);
        }
    }
    double c = a.c_sq[sys] * acc;
    const int sx = a.slot_x[lo];
    if (sx >= 0) c = fma(a.c_lin[sys], a.in_val[(size_t)sx * 1024 + lane * 33], c);
    a.out_val[(size_t)(a.uidx[lo] - a.u0) * 1024 + lane * 33] = c;
}

// FP64 masters -> FP32 hi plane and (optionally) FP32 lo plane, x = hi + lo
__global__ void k_split_f32(const double *__restrict__ v, float *__restrict__ hi, float *__restrict__ lo, int64_t n) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const double x = v[e];
    const float h = f64_to_f32(x);
    hi[e] = h;
    if (lo) lo[e] = f64_to_f32(x - f32_to_f64(h));
}


template <int B, class T>
void launch_b(const NumArgs &a, cudaStream_t st) {
    constexpr int NT = Cfg<B>::NT, LD = Cfg<B>::LD;
    size_t smem = (size_t)B * LD * sizeof(double);
    size_t ab = 2 * (size_t)B * LD * sizeof(T);
    if (ab > smem) smem = ab;
    func_smem_once((const void *)k_numeric_simt<B, T>, (int)smem);
    static int resident = 0;
    if (!resident) {
        int per_sm = 0, dev = 0, nsm = 0;
        RDM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_numeric_simt<B, T>, NT, smem));
        RDM_CUDA_TRY(cudaGetDevice(&dev));
        RDM_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        resident = std::max(1, per_sm) * nsm;
    }
    const int grid = a.max_work < resident ? a.max_work : resident;
    if (grid <= 0) return;
    k_numeric_simt<B, T><<<grid, NT, smem, st>>>(a);
    RDM_LAUNCH_CHECK();
}

// blocks of kernel k (threads per block nt, static shared memory) resident on the whole GPU
template <class K>
int resident_blocks(K k, int nt) {
    int per_sm = 0, dev = 0, nsm = 0;
    RDM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, nt, 0));
    RDM_CUDA_TRY(cudaGetDevice(&dev));
    RDM_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    return std::max(1, per_sm) * nsm;
}

template <int B, class T>
void launch_small(const NumArgs &a, cudaStream_t st) {
    static const int res = resident_blocks(k_numeric_small<B, T>, 128);
    const int per = 128 / (B * B);
    k_numeric_small<B, T><<<std::min((a.max_work + per - 1) / per, res), 128, 0, st>>>(a);
    RDM_LAUNCH_CHECK();
}

template <class T>
void dispatch(const NumArgs &a, cudaStream_t st) {
    switch (a.b) {
        case 1: launch_small<1, T>(a, st); break;
        case 2: launch_small<2, T>(a, st); break;
        case 4: launch_small<4, T>(a, st); break;
        case 8: launch_b<8, T>(a, st); break;
        case 16: launch_b<16, T>(a, st); break;
        case 32: launch_b<32, T>(a, st); break;
        case 64: launch_b<64, T>(a, st); break;
        default: throw Error{-1, "block size must be 1, 2, 4, 8, 16, 32 or 64"};
    }
}

}  // namespace

void launch_numeric_simt(const NumArgs &a, Arith ar, cudaStream_t st) {
    if (a.max_work == 0) return;
    if (ar == AR_FF) {
        if (a.b != 32 || !a.in_f32 || !a.in_f32lo) throw Error{-1, "double-FP32 products need 32 x 32 blocks"};
        static const int res = resident_blocks(k_numeric_ff_b32, 64);
        k_numeric_ff_b32<<<std::min(a.max_work, res), 64, 0, st>>>(a);
        RDM_LAUNCH_CHECK();
    } else if (ar == AR_FP64) {
        dispatch<double>(a, st);
    } else if (a.b == 32 && a.in_f32) {
        if (!a.tpos) throw Error{-1, "FP32 products of 32 x 32 blocks need the transposed positions"};
        static const int res = resident_blocks(k_numeric_f32_x2, 32);
        k_numeric_f32_x2<<<std::min(a.max_work, res), 32, 0, st>>>(a);
        RDM_LAUNCH_CHECK();
    } else {
        dispatch<float>(a, st);
    }
}

void launch_diag_fp64(const NumArgs &a, const MatSet &in, const JobTable &jt, JobMask jobs, const int *out_rp,
                      const int *out_col, const int *sys_tier, int r0, int nrows, cudaStream_t st) {
    if (nrows == 0) return;
    k_diag_fp64<<<nrows, 32, 0, st>>>(in.row_ptr.p, out_rp, out_col, a, jt, jobs, sys_tier, in.NB, r0, nrows);
    RDM_LAUNCH_CHECK();
}

void launch_to_f32(const double *val, float *f32, int64_t n, cudaStream_t st, float *f32lo) {
    if (n == 0) return;
    k_split_f32<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(val, f32, f32lo, n);
    RDM_LAUNCH_CHECK();
}

}  // namespace rdm

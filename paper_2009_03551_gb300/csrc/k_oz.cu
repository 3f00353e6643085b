// FP64-class products on the tensor cores (tcgen05 + TMEM, sm_103a) for
// 32 x 32 blocks, by exact slice products: the splitting of Ozaki, Ogita,
// Oishi and Rump (Numer. Algorithms 59, 2012), in which a matrix is cut into
// slices whose products a low-precision matrix multiply computes without
// rounding, and the slice products are summed in higher precision.  Used for
// X0^2 in the final tier of the precision ladder (S = 7 slices) and for the
// products of truncated FP64 solves (S = 8), where it takes the place of FMA
// chains on the FP64 pipe (2 FMAs per clock and SM here, 1.18 TFLOP/s in the
// CUDA-core kernel).
//
// Slices.  Row r of a matrix of the input set is scaled by sigma_r = 2^e_r,
// e_r the smallest exponent with max_k |X_rk| < 2^e_r, and x = X_rk / sigma_r in
// (-1, 1) is written in S integer digits, every one exact in bf16:
//   S = 8: base 256, x = sum_i a_i 2^-(8 i - 2) rounded at 2^-62,
//          a_i in [-128, 127] (the first one in [-64, 64]);
//   S = 7: base 128, x = sum_i a_i 2^-7i rounded at 2^-49, |a_i| <= 64 (the first
//          one 128), each digit the round-half-even of what the previous left.
// The operands are symmetric, so the slices of row c serve as the B operand of
// output column c as well (B rows = output columns, K-major), with the column
// scale sigma_c.
//
// Exact groups.  C_rc = sum_k A_rk B_kc = sigma_r sigma_c sum_g w_g D_g[r, c],
// w_g = 2^-(8 g - 4) or 2^-7g, D_g = sum_{i + j = g} sum_k a_i[r, k] b_j[c, k].
// Slice pairs with i + j <= S + 1 are kept.  Per k a group adds at most S 2^14,
// so over a segment of 128 K D_g stays within 2^24: each group accumulates in
// its own FP32 tensor-memory accumulator WITHOUT rounding (integers up to 2^24
// are exact).  Error of the 8-slice products against exact sums, largest
// element over the largest result (uniform, normal and decaying entries, one
// and two terms, 3 to 96 blocks deep): 5e-17 to 1.6e-16, that of the FP64 FMA
// chains on the same operands 4e-16 to 9e-15; in the Frobenius norm 4e-17 to
// 1e-16 against 3e-16 to 3e-15.  That error is absolute: an element below 2^-9 of
// its row's largest keeps fewer than 53 bits.  X0^2 of a 100-atom cluster, largest
// error of a block over the block's own norm: 9e-16 for norms above 0.1, 2.3e-14
// above 1e-3, 2.5e-11 above 1e-7, where FMA chains have 9e-16 throughout; the
// filter (tau >= 1e-10) drops blocks of such norms.  (7 slices: up to 2e-13 by the test's bound.)
//
// MMAs.  The accumulators of a block column lie side by side, 32 columns per
// group, and the slices of a B block one after another in shared memory, so
// one MMA multiplies slice i of A with the slices 1 .. S + 1 - i of a B block:
// N = 32 (S + 1 - i), into the groups i + 1 .. S + 1.  That is S MMAs per K = 16
// and block column instead of one per slice pair (28 of N = 64 for S = 7): an
// MMA reads its A operand (4 KB) from shared memory again, and at N = 64 those
// reads, 192 bytes per clock of MMA where shared memory delivers 128, bounded
// the kernel.  X0^2 of the final tier, 2,000-atom cluster in the bf16 ladder:
// 27.5 -> 22.1 ms per solve.
//
// Tiles are 128 x 64: 4 block rows (one MMA operand) x 2 block columns, whose
// accumulators (S x 32 columns each) are separate: the last K-step of a
// segment finishes block column 0 half a step before block column 1, and the
// next segment's first K-step starts with block column 0, so that each of the
// two is drained by its four epilogue warps while the MMAs of the other run.
// (Running both last steps' block column 0 before their block column 1, to hide
// more of the draining, holds both stages longer and exposes their refill:
// 19.1 -> 23.0 ms per solve of the 2,000-atom cluster.)  Tiles are handed out by
// an atomic counter (round robin: 22.2 ms): the copy warp claims the next one
// after the first copies of this one.
//
// Epilogue, S = 8.  The group sums are integers and are added up as integers,
// four groups at a time in 64-bit words (units 2^-36 and 2^-68), converted
// from FP32 by adding 1.5 * 2^23 (exact for |D| <= 2^22; larger sums, which take
// operands whose digits are nearly all extreme, are detected and converted one
// by one).  The sum is therefore exact and does not depend on how the K-steps
// are cut into tiles and segments.  It is rounded to FP64 once, in integer
// arithmetic (8,192 conversions per tile on the FP64 pipe would take as long
// as a K-step's MMAs).  S = 7: the groups are added, largest first, to a
// double-FP32 sum by Knuth's TwoSum (about 48 bits).  With two terms
// (A B + B A) the first one's sum goes to the output slot and is added in
// FP64 to the second's.  Then C = c_lin X + c_sq P in FP64, Frobenius norm (for
// S = 8 in FP32, and in FP64 where that lies within 1e-5 of the threshold),
// truncation flag, FP64 store.  Diagonal blocks come out exactly symmetric:
// (r, c) and (c, r) have the same sums, in the other order for two terms, and
// FP64 addition commutes.
//
// Operands.  A K-step brings 4 A blocks and 2 B blocks of S bf16 slices (96 KB
// for S = 8) for 128 x 64 x 32 FP64-class multiply-adds.  A block needs its 8-row
// groups equally spaced over the 4 stacked blocks (groups outermost, slices
// inside) and B its slices (slices outermost), so both layouts are stored.
// FP64 solve of a 300-atom cluster: products 652 ms on the FP64 pipe, 33 ms here
// (24 TFLOP/s useful, the 2 ms of k_diag_fp64 included: the diagonal elements
// of X0^2 keep the FMA chains' rounding, because the trace decides branches).  Bounded waits and the abort drain are those of the
// split kernel (k_tc.cu).  ptxas: 162 registers for S = 7; 168, the bound of its
// launch, and 196 bytes of spills for S = 8.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "fp_bits.cuh"
#include "tc_gemm.cuh"
#include "tc_plan.cuh"
#include "tc_ptx.cuh"

namespace rdm {
namespace {

// S slices per element, groups g = i + j = 2 .. S + 1
template <int S>
struct GeoOz : PlanGeo<4, 2> {
    static constexpr int kSliceElems = 32 * 32;
    static constexpr int kBlockElems = S * kSliceElems;             // one layout of a block's slices
    static constexpr int kBlockBytes = 2 * kBlockElems;             // 16 KB (S = 8)
    static constexpr int kSideABytes = TBM * kBlockBytes;
    static constexpr int kStageBytes = kSlots * kBlockBytes;        // 96 KB
    static constexpr int kStages = 2;
    static constexpr int kSegSteps = 4;                             // K-steps per segment: 128 K
    static constexpr uint32_t kSBOA = S * 512;                      // bytes between 8-row groups of an A slice
    static constexpr uint32_t kSBOB = 512;                          // ... of a B slice, and on to the next slice
    static constexpr int kAccCols = 32 * S;                         // accumulator columns of a block column
    static_assert(2 * kAccCols <= 512, "group accumulators exceed tensor memory");
};
constexpr int kOzEpiWarp0 = 2, kOzEpiWarps = 8;
constexpr int kOzThreads = 32 * (kOzEpiWarp0 + kOzEpiWarps);
constexpr int kOzBadRow = 1 << 20;      // exponent of a row with infinities or NaN: its products are NaN

// element (r, c), slice i of a block.  A layout: the 8-row groups of the
// slices alternate (512 bytes each); B layout: slice after slice.  Inside a
// group, core matrix (c / 8) at 64 elements.
template <int S>
__device__ __forceinline__ int oz_offset_a(int r, int c, int i) {
    return (r >> 3) * (S * 256) + i * 256 + ((c >> 3) << 6) + ((r & 7) << 3) + (c & 7);
}
__device__ __forceinline__ int oz_offset_b(int r, int c, int i) {
    return i * 1024 + (r >> 3) * 256 + ((c >> 3) << 6) + ((r & 7) << 3) + (c & 7);
}

// e_r of every row of `nrows` flat block rows, from the exponent fields of the
// elements (integer maxima: FP64 comparisons run on the FP64 pipe): one block
// row per CTA, 8 threads per row; and the flat block row of every block
__global__ void __launch_bounds__(256) k_oz_row_exp(const int *__restrict__ row_ptr, const double *__restrict__ val,
                                                     int nrows, int *__restrict__ e, int *__restrict__ row_of) {
    const int i = blockIdx.x;
    if (i >= nrows) return;
    const int r = threadIdx.x >> 3, q = threadIdx.x & 7;   // row r of the block row, columns 4q .. 4q + 3
    const int p0 = row_ptr[i], p1 = row_ptr[i + 1];
    for (int p = p0 + threadIdx.x; p < p1; p += 256) row_of[p] = i;
    int mx = 0;
    for (int p = p0; p < p1; ++p) {
        const int4 *v = reinterpret_cast<const int4 *>(val + (size_t)p * 1024 + r * 32 + 4 * q);
        const int4 v0 = v[0], v1 = v[1];                   // high words: y and w
        mx = max(mx, max(max(v0.y & 0x7fffffff, v0.w & 0x7fffffff), max(v1.y & 0x7fffffff, v1.w & 0x7fffffff)));
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const int E = mx >> 20;
    if (q == 0) e[(size_t)i * 32 + r] = E == 0x7ff ? kOzBadRow : E > 0 ? E - 1022 : 0;
}

// The 7 base-128 digits of x0 = v 2^-er (|x0| < 1: 2^er bounds the
// row), each the round-half-even of the remainder times 128, as in the
// slicing of Ozaki, Ogita, Oishi and Rump: x0 = sum_i a_i 2^(-7(i+1)) + a
// remainder below 2^-49.  Integer arithmetic, exact (FP64 throughput is low
// on this part): X = x0 2^60 is held as its floor plus a sticky bit for the
// bits below; digit i has unit 2^(53 - 7i) in X.
__device__ __forceinline__ void oz_digits(double v, int er, int (&a)[7]) {
    const uint64_t bits = (uint64_t)__double_as_longlong(v);
    const bool neg = (bits >> 63) != 0;
    const int E = (int)((bits >> 52) & 0x7FF);
    uint64_t M = bits & ((1ull << 52) - 1);
    int ex = 1 - 1075;                                   // subnormal
    if (E != 0) {
        M |= 1ull << 52;
        ex = E - 1075;
    }
    const int sh = ex - er + 60;                         // |x0| 2^60 = M 2^sh
    int64_t X = 0;
    bool sticky = false;
    if (M != 0) {
        if (sh >= 0) {
            X = (int64_t)(M << sh);                      // sh <= 7: M 2^sh < 2^60
        } else {
            const int rs = -sh;
            const uint64_t q = rs >= 64 ? 0ull : M >> rs;
            sticky = rs >= 64 ? true : (M & ((1ull << rs) - 1)) != 0;
            X = (int64_t)q;
        }
        if (neg) X = -X - (sticky ? 1 : 0);              // the floor of the negative value
    }
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const int s = 53 - 7 * i;
        int64_t q = X >> s;                              // floor
        const int64_t r = X - (q << s);                  // in [0, 2^s); true fraction (r + sticky) / 2^s
        const int64_t half = 1ll << (s - 1);
        if (r > half || (r == half && (sticky || (q & 1)))) q += 1;
        a[i] = (int)q;
        X -= q << s;
    }
}

// x 2^(62 - er) rounded to an integer, for |x| < 2^er (0 in a bad row)
__device__ __forceinline__ int64_t oz_fixed(double v, int er) {
    const uint64_t bits = (uint64_t)__double_as_longlong(v);
    const int E = (int)((bits >> 52) & 0x7FF);
    uint64_t M = bits & ((1ull << 52) - 1);
    if (E != 0) M |= 1ull << 52;
    const int sh = (E != 0 ? E : 1) - 1075 - er + 62;      // the value is M 2^sh
    uint64_t q = 0;
    if (sh >= 0) q = M << (sh & 63);                              // below 2^62
    else if (sh > -64) q = ((M >> (-sh - 1)) + 1) >> 1;
    if (er == kOzBadRow) q = 0;
    return (bits >> 63) ? -(int64_t)q : (int64_t)q;
}

// Slices of the blocks of the set, in both layouts: one thread per 8
// consecutive elements of a block row.  S = 8: with 128 added to every digit
// but the first, the digits are the bytes of the sum; a byte placed in the
// fraction of 2^23 is converted to FP32 by subtracting 2^23 + 128.  The top
// half of the FP32 value of a digit is its bf16 value.
template <int S>
__global__ void k_oz_slices(const double *__restrict__ val, const int *__restrict__ row_of,
                            const int *__restrict__ e, int64_t nblk, uint16_t *__restrict__ out_a,
                            uint16_t *__restrict__ out_b) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= nblk * 128) return;
    const int64_t p = g >> 7;
    const int rc0 = (int)(g & 127) * 8;
    const int r = rc0 >> 5, c0 = rc0 & 31;
    const int er = e[(size_t)row_of[p] * 32 + r];
    const double2 *v2 = reinterpret_cast<const double2 *>(val + p * 1024 + rc0);
    double2 x2[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x2[k] = v2[k];
    uint32_t h[S][8];       // FP32 values of the digits
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const double x = k & 1 ? x2[k >> 1].y : x2[k >> 1].x;
        if constexpr (S == 8) {
            const uint64_t y = (uint64_t)oz_fixed(x, er) + 0x0080808080808080ull;
            const uint32_t lo = (uint32_t)y, hi = (uint32_t)(y >> 32);
            h[0][k] = __float_as_uint(__int_as_float(0x4B400000 + ((int)hi >> 24)) - 12582912.0f);   // signed
#pragma unroll
            for (int i = 1; i < 8; ++i)
                h[i][k] = __float_as_uint(
                    __uint_as_float(__byte_perm(7 - i < 4 ? lo : hi, 0x4B000000u, 0x7440 + ((7 - i) & 3))) - 8388736.0f);
        } else {
            int a[7];
            oz_digits(x, er, a);
#pragma unroll
            for (int i = 0; i < 7; ++i)
                h[i][k] = __float_as_uint(__int_as_float(0x4B400000 + a[i]) - 12582912.0f);
        }
    }
#pragma unroll
    for (int i = 0; i < S; ++i) {
        uint4 o;
        o.x = __byte_perm(h[i][0], h[i][1], 0x7632); o.y = __byte_perm(h[i][2], h[i][3], 0x7632);
        o.z = __byte_perm(h[i][4], h[i][5], 0x7632); o.w = __byte_perm(h[i][6], h[i][7], 0x7632);
        *reinterpret_cast<uint4 *>(out_a + p * (S * 1024) + oz_offset_a<S>(r, c0, i)) = o;
        *reinterpret_cast<uint4 *>(out_b + p * (S * 1024) + oz_offset_b(r, c0, i)) = o;
    }
}

// ---------------------------------------------------------------------------
// sums of the groups and their conversion
// ---------------------------------------------------------------------------
constexpr int kMagicBits = 0x4B400000;               // 1.5 * 2^23

// the integers (int)p[0] 256 + (int)p[1], exact for |p| <= 2^22
__device__ __forceinline__ int oz_pair(float p0, float p1) {
    const int b0 = __float_as_int(p0 + 12582912.0f), b1 = __float_as_int(p1 + 12582912.0f);
    return (int)((uint32_t)b0 * 256u + (uint32_t)b1 - (uint32_t)kMagicBits * 257u);
}

// hi 2^-36 + lo 2^-68, rounded to nearest even and scaled by 2^ex
__device__ __forceinline__ double oz_to_f64(int64_t hi, int64_t lo, int ex) {
    hi += lo >> 32;
    uint32_t l = (uint32_t)lo;                                   // the fraction of hi, 32 bits
    const bool neg = hi < 0;
    uint64_t m = (uint64_t)hi;
    if (neg) {
        m = ~m + (l == 0u ? 1u : 0u);
        l = 0u - l;
    }
    int E = 1023 + 63 - 36 + ex;
    if (m == 0) {                                                // below one unit of hi
        m = (uint64_t)l << 32;
        l = 0u;
        E -= 64;
        if (m == 0) return 0.0;
    }
    const int n = __clzll((long long)m);
    if (n) m = (m << n) | (((uint64_t)l << 32) >> (64 - n));
    E -= n;
    uint64_t r = m >> 11;
    r += (((uint32_t)m & 0x7ffu) + ((uint32_t)r & 1u)) > 0x400u ? 1u : 0u;
    if (E < 1 || E > 2045) {                                     // outside the normal range
        const double v = ldexp((double)r, E - 1075);
        return neg ? -v : v;
    }
    r += (uint64_t)(E - 1) << 52;
    return __longlong_as_double((long long)(r | (neg ? 1ull << 63 : 0ull)));
}

// x added to (hi, lo) by Knuth's TwoSum (exact sum hi + x = s + t), the
// rounding error t carried in lo
__device__ __forceinline__ void ff_add(float &hi, float &lo, float x) {
    const float s = __fadd_rn(hi, x);
    const float bp = __fsub_rn(s, hi);
    const float t = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
    hi = s;
    lo = __fadd_rn(lo, t);
}

// v 2^ex (the exponent field while the result is normal)
__device__ __forceinline__ double scale_pow2(double v, int ex) {
    const int hi = __double2hiint(v);
    const int E = (hi >> 20) & 0x7ff;
    if (E == 0 || E == 0x7ff || E + ex < 1 || E + ex > 2046) return ldexp(v, ex);
    return __hiloint2double(hi + ex * 1048576, __double2loint(v));
}

struct OzArgs {
    const uint16_t *slices_a, *slices_b;   // slices of the operand matrices' blocks, both layouts
    const uint16_t *zero;         // zero blocks (kSlots per CTA)
    const int *e;                 // row exponents (flat rows of the set)
    const int *tiles;
    const int64_t *step_rng;
    const int *steps;
    const int *flags;             // TcWork::counters
    int *next_tile;               // tiles handed out beyond every CTA's first
    int NB;
    // epilogue
    const double *in_val;
    const int *slot_row, *slot_job, *slot_x;
    const int *mcol;
    const int *sys_of_row;
    const double *c_lin, *c_sq, *tau0, *tau1;
    int job_tau_sel[kMaxJobs], job_nterm[kMaxJobs], job_a[kMaxJobs][2], job_b[kMaxJobs][2];
    double *out_val;
    float *out_nrm;
    uint8_t *keep;
    const int *uidx;
    int64_t u0;
    int *err;
    long long wait_cycles;
};

struct __align__(16) OzCtl {
    TileSeq seq;
    uint64_t full[2], empty[2];
    uint64_t seg_full[2], seg_empty[2];      // per block column of the tile
    uint64_t drain;
    uint32_t tmem_base;
    int abort_flag;
};

// segments of a tile: the K-steps of the first term, then those of the second
// (which has other scales), kSegSteps at a time
__device__ __forceinline__ int oz_segments(int steps) { return (steps + 3) / 4; }

template <int S>
__global__ void __launch_bounds__(kOzThreads, 1) k_tc_oz(OzArgs A) {
    using G = GeoOz<S>;
    static_assert(G::kSegSteps == 4 && G::kStages == 2, "oz_segments, OzCtl");
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *stages = smem_raw;
    OzCtl *ctl = reinterpret_cast<OzCtl *>(smem_raw + G::kStages * G::kStageBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int *abort_flag = &ctl->abort_flag;
    if (A.flags[1]) return;               // the K-step list outgrew its buffer: the host builds it again
    const int ntile = A.flags[2];

    if (threadIdx.x == 0) {
        for (int s = 0; s < G::kStages; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&ctl->seg_full[b], 1); mbar_init(&ctl->seg_empty[b], kOzEpiWarps / 2); }
        init_seq(&ctl->seq, 2 + kOzEpiWarps);
        mbar_init(&ctl->drain, 1);
        ctl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&ctl->tmem_base)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = ctl->tmem_base;

    if (warp == 0) {
        // ---------------- producer: one bulk copy per operand block ----------------
        uint32_t it = 0;
        bool ok = true;
        uint32_t zmask[G::kStages];
#pragma unroll
        for (int k = 0; k < G::kStages; ++k) zmask[k] = 0u;
        const uint16_t *base = lane < G::TBM ? A.slices_a : A.slices_b;
        // lane 0 claims the CTA's next tile once the first copies of this one are issued
        TileEntry e{};
        uint32_t k = 0;
        auto claim = [&]() {
            if (lane == 0) put_tile(&ctl->seq, k, ntile, A.step_rng, A.next_tile, abort_flag, A.wait_cycles);
            __syncwarp();
        };
        claim();
        while (ok && take_tile<32>(&ctl->seq, k, lane, abort_flag, A.wait_cycles, e) && e.t < ntile) {
            const int64_t s0 = e.s0, s1 = e.s1;
            ++k;
            if (s0 == s1) claim();
            int nxt = (s0 < s1 && lane < G::kSlots) ? A.steps[s0 * G::kSlots + lane] : -1;
            for (int64_t q = s0; q < s1; ++q, ++it) {
                const int cur = nxt;
                if (q + 1 < s1 && lane < G::kSlots) nxt = A.steps[(q + 1) * G::kSlots + lane];
                const int st = it % G::kStages;
                const uint32_t ph = (it / G::kStages) & 1;
                const uint32_t zbits = __ballot_sync(0xffffffffu, lane < G::kSlots && cur < 0);
                uint32_t zprev = 0u;
#pragma unroll
                for (int k = 0; k < G::kStages; ++k)
                    if (k == st) {
                        zprev = zmask[k];
                        zmask[k] = zbits;
                    }
                const bool skip = lane >= G::kSlots || (cur < 0 && ((zprev >> lane) & 1u));
                const uint32_t need = __ballot_sync(0xffffffffu, !skip);
                int waited = 1;
                if (lane == 0) {
                    waited = mbar_wait(&ctl->empty[st], ph ^ 1, abort_flag, A.wait_cycles) ? 1 : 0;
                    if (waited) mbar_expect_tx(&ctl->full[st], (uint32_t)__popc(need) * G::kBlockBytes);
                }
                waited = __shfl_sync(0xffffffffu, waited, 0);
                if (!waited) { ok = false; break; }
                if (!skip) {
                    const uint16_t *src = cur >= 0 ? base + (size_t)cur * G::kBlockElems
                                                   : A.zero + ((size_t)blockIdx.x * G::kSlots + lane) * G::kBlockElems;
                    bulk_g2s(stages + st * G::kStageBytes + lane * G::kBlockBytes, src, G::kBlockBytes, &ctl->full[st]);
                }
                if (q == s0) claim();
            }
        }
        if ((!ok || *abort_flag) && lane == 0) {
            // after an abort, wait (bounded) for the copies still in flight
            const uint32_t n = it < (uint32_t)G::kStages ? it : (uint32_t)G::kStages;
            for (uint32_t q = it - n; q < it; ++q)
                mbar_wait_drain(&ctl->full[q % G::kStages], (q / G::kStages) & 1, A.wait_cycles);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            // kind::f16: D = F32, A = B = BF16, K-major, M = 128; N is added below
            const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);
            uint32_t it = 0, seg = 0;
            bool issued = false;
            TileEntry e{};
            for (uint32_t k = 0; take_tile<1>(&ctl->seq, k, 0, abort_flag, A.wait_cycles, e) && e.t < ntile; ++k) {
                const int *d = A.tiles + (size_t)e.t * G::kTileInts;
                const int nst = d[3], n1 = d[2];
                bool ok = true;
                for (int q = 0; q < nst && ok; ++seg) {
                    const int end = q < n1 ? n1 : nst;
                    const int qs = q, qe = q + G::kSegSteps < end ? q + G::kSegSteps : end;
                    for (; q < qe; ++q, ++it) {
                        const int st = it % G::kStages;
                        const uint32_t ph = (it / G::kStages) & 1;
                        if (!mbar_wait(&ctl->full[st], ph, abort_flag, A.wait_cycles)) { ok = false; break; }
                        fence_after();
                        const uint32_t base = smem_u32(stages + st * G::kStageBytes);
                        for (int bc = 0; bc < 2; ++bc) {
                            if (q == qs) {
                                if (!mbar_wait(&ctl->seg_empty[bc], (seg & 1) ^ 1, abort_flag, A.wait_cycles)) { ok = false; break; }
                                fence_after();
                            }
                            const uint32_t bb = base + G::kSideABytes + bc * G::kBlockBytes;
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
                                for (int i = 0; i < S; ++i)
                                    mma_f16(tmem + bc * G::kAccCols + 32 * i,
                                            smem_desc(base + i * 512 + kk * 256, 128, G::kSBOA),
                                            smem_desc(bb + kk * 256, 128, G::kSBOB),
                                            idesc0 | ((uint32_t)(4 * (S - i)) << 17),       // N = 32 (S - i)
                                            q == qs && kk == 0 && i == 0 ? 0u : 1u);
                            }
                            issued = true;
                            if (q == qe - 1) mma_commit(&ctl->seg_full[bc]);
                        }
                        if (!ok) break;
                        mma_commit(&ctl->empty[st]);
                    }
                }
                if (!ok) break;
            }
            if (*abort_flag && issued) {
                mma_commit(&ctl->drain);
                long long t0 = clock64();
                while (!mbar_try_wait(&ctl->drain, 0) && clock64() - t0 < A.wait_cycles) {
                }
            }
        }
    } else {
        // ---------------- epilogue: warps 2..9, one 32 x 32 output block each ----------------
        const int eq = warp & 3;                        // TMEM lanes 32 eq .. 32 eq + 31: block row eq
        const int bc = (warp - kOzEpiWarp0) >> 2;       // block column of the tile
        const uint32_t ta = tmem + ((uint32_t)(32 * eq) << 16) + bc * G::kAccCols;
        uint32_t seg = 0;
        TileEntry e{};
        for (uint32_t k = 0; take_tile<32>(&ctl->seq, k, lane, abort_flag, A.wait_cycles, e) && e.t < ntile; ++k) {
            const int *d = A.tiles + (size_t)e.t * G::kTileInts;
            const int s = d[4 + eq * G::TBN + bc];
            const int nst = d[3], n1 = d[2];
            if ((nst < 0 || n1 < 0 || n1 > nst) && lane == 0) atomicOr(A.err, 4);
            int job = 0, i = 0, j = 0, sys = 0;
            if (s >= 0) {
                i = A.slot_row[s];
                j = A.mcol[s];
                job = A.slot_job[s];
                sys = A.sys_of_row[i];
            }
            double *o = s >= 0 ? A.out_val + (size_t)(A.uidx[s] - (int)A.u0) * 1024 + lane * 32 : nullptr;
            const int nterm = s >= 0 ? A.job_nterm[job] : 2;
            bool ok = true;
            for (int term = 0; term < 2 && ok; ++term) {
                const int nseg = nst > 0 ? oz_segments(term == 0 ? n1 : nst - n1) : 0;
                // sums of the groups: integers (S = 8) or double-FP32 (S = 7)
                using Sum = typename std::conditional<S == 8, int64_t, float>::type;
                Sum hi[32], lo[32];
#pragma unroll
                for (int c = 0; c < 32; ++c) hi[c] = lo[c] = 0;
                for (int g = 0; g < nseg; ++g, ++seg) {
                    if (!mbar_wait(&ctl->seg_full[bc], seg & 1, abort_flag, A.wait_cycles)) { ok = false; break; }
                    fence_after();
#pragma unroll
                    for (int c0 = 0; c0 < 32; c0 += 8) {
#pragma unroll
                        for (int half = 0; half < 2; ++half) {
                            float p[4][8];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                if (4 * half + u < S) {
                                    tmem_ld8(ta + (4 * half + u) * 32 + c0, p[u]);
                                } else {
#pragma unroll
                                    for (int c = 0; c < 8; ++c) p[u][c] = 0.f;
                                }
                            }
                            tmem_wait_ld(p);
                            if constexpr (S == 8) {
                                float mx = 0.f;
#pragma unroll
                                for (int u = 0; u < 4; ++u)
#pragma unroll
                                    for (int c = 0; c < 8; ++c) mx = fmaxf(mx, fabsf(p[u][c]));
                                Sum(&w)[32] = half == 0 ? hi : lo;
                                if (mx <= 4194304.0f) {
#pragma unroll
                                    for (int c = 0; c < 8; ++c) {
                                        w[c0 + c] += (int64_t)oz_pair(p[0][c], p[1][c]) * 65536;
                                        w[c0 + c] += oz_pair(p[2][c], p[3][c]);
                                    }
                                } else {
                                    // sums beyond 2^22
#pragma unroll
                                    for (int c = 0; c < 8; ++c)
                                        w[c0 + c] += (((int64_t)p[0][c] * 256 + (int64_t)p[1][c]) * 256 + (int64_t)p[2][c]) * 256 +
                                                     (int64_t)p[3][c];
                                }
                            } else {
                                // largest first, scaled by 2^(-7 g)
#pragma unroll
                                for (int u = 0; u < 4; ++u)
                                    if (4 * half + u < S) {
                                        const float sc = __int_as_float((127 - 7 * (4 * half + u + 2)) << 23);
#pragma unroll
                                        for (int c = 0; c < 8; ++c) ff_add(hi[c0 + c], lo[c0 + c], p[u][c] * sc);
                                    }
                            }
                        }
                    }
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ctl->seg_empty[bc]);
                }
                if (!ok || s < 0 || term >= nterm) continue;
                // P = sigma_r sigma_c (sum of the groups)
                const int er = A.e[((size_t)A.job_a[job][term] * A.NB + i) * 32 + lane];
                const int ec_l = A.e[((size_t)A.job_b[job][term] * A.NB + j) * 32 + lane];
                const bool last = term == nterm - 1;
                const double cl = A.c_lin[sys], cq = A.c_sq[sys];
                const double tau = A.job_tau_sel[job] ? A.tau1[sys] : A.tau0[sys];
                const int sx = A.slot_x[s];
                const double *gx = (last && sx >= 0 && cl != 0.0) ? A.in_val + (size_t)sx * 1024 + lane * 32 : nullptr;
                float ss = 0.f;
                double s2 = 0.0;
#pragma unroll
                for (int c4 = 0; c4 < 32; c4 += 4) {
                    double xo[4] = {0.0, 0.0, 0.0, 0.0}, po[4] = {0.0, 0.0, 0.0, 0.0}, r[4];
                    if (gx) ld_f64x4(gx + c4, xo);
                    if (term == 1) ld_f64x4(o + c4, po);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int c = c4 + u;
                        const int ec = __shfl_sync(0xffffffffu, ec_l, c);
                        double p;
                        if constexpr (S == 8) p = oz_to_f64(hi[c], lo[c], er + ec);
                        else p = scale_pow2(f32_to_f64(hi[c]) + f32_to_f64(lo[c]), er + ec);
                        if (er == kOzBadRow || ec == kOzBadRow) p = __longlong_as_double(0x7ff8000000000000ll);
                        if (term == 1) p += po[u];
                        r[u] = !last ? p : gx ? fma(cl, xo[u], cq == 1.0 ? p : cq * p) : cq == 1.0 ? p : cq * p;
                    }
                    st_f64x4(o + c4, r);
                    if (!last) continue;
                    if constexpr (S == 8) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float f = f64_to_f32(r[u]);
                            ss = fmaf(f, f, ss);
                        }
                    } else {
                        s2 = fma(r[0], r[0], fma(r[1], r[1], s2));
                        s2 = fma(r[2], r[2], fma(r[3], r[3], s2));
                    }
                }
                if (!last) continue;
                float nrm;
                bool kp;
                if constexpr (S == 8) {
#pragma unroll
                    for (int w = 16; w > 0; w >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, w);
                    nrm = sqrtf(ss) * (1.0f + 4e-6f);
                    kp = (double)nrm >= tau && nrm > 0.f;
                    // near the threshold, or where FP32 squares leave the range, the FP64 norm decides
                    if (!(fabs((double)nrm - tau) > 1e-5 * tau) || ss < 1e-30f || !(ss < 1e30f)) {
                        for (int c = 0; c < 32; ++c) s2 = fma(o[c], o[c], s2);
#pragma unroll
                        for (int w = 16; w > 0; w >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, w);
                        const double n2 = sqrt(s2);
                        nrm = __double2float_ru(n2);
                        kp = n2 >= tau && n2 > 0.0;
                    }
                } else {
#pragma unroll
                    for (int w = 16; w > 0; w >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, w);
                    nrm = __double2float_ru(sqrt(s2)) * (1.0f + 1e-6f);
                    kp = (double)nrm >= tau && nrm > 0.f;
                }
                if (lane == 0) {
                    A.out_nrm[s] = nrm;
                    A.keep[s] = kp ? kKeepBlock : 0;
                }
            }
            if (!ok) break;
        }
    }

    fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && ctl->abort_flag) atomicOr(A.err, 1);
    if (warp == 1) {
        __syncwarp();
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

template <int S>
constexpr size_t oz_smem() { return (size_t)GeoOz<S>::kStages * GeoOz<S>::kStageBytes + sizeof(OzCtl); }
static_assert(oz_smem<8>() <= 227 * 1024, "shared memory of the slice-product kernel exceeds 227 KB");

template <int S>
void launch_oz(OzArgs &A, const TcPlan &plan, OzWork &ow, cudaStream_t st) {
    using G = GeoOz<S>;
    int dev = 0, nsm = 0;
    RDM_CUDA_TRY(cudaGetDevice(&dev));
    RDM_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const size_t zero_elems = (size_t)nsm * G::kSlots * G::kBlockElems;
    if (!ow.zero.p || ow.zero.cap < zero_elems) {
        ow.zero.ensure(zero_elems);
        RDM_CUDA_TRY(cudaMemsetAsync(ow.zero.p, 0, ow.zero.cap * sizeof(uint16_t), st));
    }
    A.zero = ow.zero.p;
    func_smem_once((const void *)k_tc_oz<S>, (int)oz_smem<S>());
    const int grid = plan.max_tile < nsm ? plan.max_tile : nsm;
    k_tc_oz<S><<<grid, kOzThreads, oz_smem<S>(), st>>>(A);
    RDM_LAUNCH_CHECK();
}

}  // namespace

bool prepare_oz_operands(const MatSet &in, int nmat, int slices, size_t reserve, OzWork &w, cudaStream_t st) {
    if (in.b != 32) throw Error{-1, "the slice-product (FP64-class tensor-core) path handles 32 x 32 blocks"};
    const int nrows = nmat * in.NB;
    int64_t nblk = 0;
    for (int m = 0; m < nmat; ++m) nblk += in.nnzb[m];
    const size_t elems = (size_t)std::max<int64_t>(nblk, 1) * slices * 1024;
    if (w.slices_a.cap < elems || w.slices_b.cap < elems) {
        // room for both layouts (and their headroom), or the caller's other path
        size_t fr = 0, tot = 0;
        RDM_CUDA_TRY(cudaMemGetInfo(&fr, &tot));
        const size_t need = 4 * DevBuf<uint16_t>::with_headroom(elems) + reserve;   // 2 layouts x 2 bytes
        if (need > fr + (w.slices_a.cap + w.slices_b.cap) * sizeof(uint16_t)) return false;
    }
    w.nslice = slices;
    w.e.ensure((size_t)std::max(nrows, 1) * 32);
    w.row_of.ensure(std::max<int64_t>(nblk, 1));
    w.slices_a.ensure(elems);
    w.slices_b.ensure(elems);
    if (nrows == 0) return true;
    k_oz_row_exp<<<nrows, 256, 0, st>>>(in.row_ptr.p, in.val.p, nrows, w.e.p, w.row_of.p);
    RDM_LAUNCH_CHECK();
    if (nblk == 0) return true;
    const unsigned grid = (unsigned)((nblk * 128 + 255) / 256);
    if (slices == 8)
        k_oz_slices<8><<<grid, 256, 0, st>>>(in.val.p, w.row_of.p, w.e.p, nblk, w.slices_a.p, w.slices_b.p);
    else
        k_oz_slices<7><<<grid, 256, 0, st>>>(in.val.p, w.row_of.p, w.e.p, nblk, w.slices_a.p, w.slices_b.p);
    RDM_LAUNCH_CHECK();
    return true;
}

TcPlan build_oz_plan(const MatSet &in, const JobTable &jt, const SysDev &sd, const int *out_rp, const int *mcol,
                     TcWork &w, JobMask job_mask, int unit0, int unit1, int64_t nupper, int64_t min_steps,
                     cudaStream_t st) {
    if (in.b != 32) throw Error{-1, "the slice-product (FP64-class tensor-core) path handles 32 x 32 blocks"};
    return build_plan<GeoOz<8>>(in, jt, sd, out_rp, mcol, w, job_mask, unit0, unit1, nupper, min_steps, st);
}

double oz_step_flops(const OzWork &ow) { return ow.nslice * (ow.nslice + 1) / 2 * 2.0 * 2.0 * 128.0 * 64.0 * 16.0; }

void launch_numeric_oz(const NumArgs &a, const MatSet &in, const JobTable &jt, const int *mcol, OzWork &ow,
                         TcWork &w, const TcPlan &plan, cudaStream_t st) {
    if (plan.max_tile == 0) return;
    OzArgs A{};
    A.slices_a = ow.slices_a.p;
    A.slices_b = ow.slices_b.p;
    A.e = ow.e.p;
    A.NB = in.NB;
    A.tiles = w.tiles.p; A.step_rng = w.step_rng.p; A.steps = w.steps.p; A.flags = w.counters;
    A.in_val = a.in_val; A.slot_row = a.slot_row; A.slot_job = a.slot_job; A.slot_x = a.slot_x; A.mcol = mcol;
    A.sys_of_row = a.sys_of_row; A.c_lin = a.c_lin; A.c_sq = a.c_sq; A.tau0 = a.tau0; A.tau1 = a.tau1;
    for (int p = 0; p < kMaxJobs; ++p) A.job_tau_sel[p] = a.job_tau_sel[p];
    for (int p = 0; p < jt.njob; ++p) {
        A.job_nterm[p] = jt.job[p].nterm;
        for (int t = 0; t < 2; ++t) {
            A.job_a[p][t] = jt.job[p].a[t];
            A.job_b[p][t] = jt.job[p].b[t];
        }
    }
    A.out_val = a.out_val; A.out_nrm = a.out_nrm; A.keep = a.keep; A.uidx = a.uidx; A.u0 = a.u0;
    A.err = w.counters;
    A.next_tile = w.counters + 6;
    A.wait_cycles = w.knobs.wait_cycles > 0 ? w.knobs.wait_cycles : kWaitCycles;
    if (ow.nslice == 8) launch_oz<8>(A, plan, ow, st);
    else launch_oz<7>(A, plan, ow, st);
}

}  // namespace rdm

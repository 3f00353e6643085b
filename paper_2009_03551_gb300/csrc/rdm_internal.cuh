// Internal declarations of the GB300 response-density-matrix library.
//
// Data model
// ----------
// A batch of independent systems is stored as ONE block-diagonal block-sparse
// matrix over NB = sum_s nb_s block rows; system s owns block rows (and block
// columns) [row0[s], row0[s] + nb[s]).  All systems share the block size b.
//
// A MatSet holds nmat such matrices over the same block-row space, in one set
// of arrays: blocks of matrix m occupy global block indices
// [row_ptr[m*NB], row_ptr[m*NB+NB]) (row_ptr has nmat*NB+1 entries, so row i
// of matrix m is [row_ptr[m*NB+i], row_ptr[m*NB+i+1])).  row_ptr entries are global
// block indices; col_idx holds global block columns (sorted inside a row);
// val holds b*b FP64 values per block (row-major); nrm holds an FP32 upper
// bound of every block's Frobenius norm.  In the solve, matrix 0 is X0 and
// matrices 1..nd are X1_gamma.  Patterns of every matrix are symmetric and
// values are symmetric (block (j,i) is the transpose of block (i,j)).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <atomic>
#include <string>
#include <utility>
#include <vector>

namespace rdm {

// ---------------------------------------------------------------------------
// error handling inside the library (converted to status codes at the ABI)
// ---------------------------------------------------------------------------
struct Error {
    int code;
    std::string msg;
};

#define RDM_CUDA_TRY(expr)                                                        \
    do {                                                                          \
        cudaError_t _e = (expr);                                                  \
        if (_e != cudaSuccess)                                                    \
            throw ::rdm::Error{_e == cudaErrorMemoryAllocation ? -3 : -4,         \
                               std::string(#expr) + ": " + cudaGetErrorString(_e)}; \
    } while (0)

// every kernel launch of the library goes through RDM_LAUNCH_CHECK, which
// also counts it (the count is reported per solve in rdm_info)
extern thread_local long long g_kernel_launches;   // launches of this thread (a solve runs on one thread)
#define RDM_LAUNCH_CHECK()                      \
    do {                                        \
        ++::rdm::g_kernel_launches;             \
        RDM_CUDA_TRY(cudaGetLastError());       \
    } while (0)

// cudaFuncAttributeMaxDynamicSharedMemorySize of kernel `func`, set once per
// kernel and device (the attribute is per device; handles of one process may
// use several, and solves may run on worker threads)
void func_smem_once(const void *func, int bytes);

// device bytes held by all DevBufs of the process (current and high-water mark)
inline std::atomic<size_t> g_dev_bytes{0};
inline std::atomic<size_t> g_dev_bytes_peak{0};

// test setting: > 0: the g_fail_alloc-th allocation of this thread from now on fails
inline thread_local int g_fail_alloc = 0;

inline void *dev_alloc(size_t bytes) {
    void *p = nullptr;
    cudaError_t e = g_fail_alloc > 0 && --g_fail_alloc == 0 ? cudaErrorMemoryAllocation : cudaMalloc(&p, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        throw Error{-3, "cudaMalloc of " + std::to_string(bytes) + " bytes failed (" +
                            std::to_string(g_dev_bytes.load()) + " bytes held by the library)"};
    }
    const size_t now = g_dev_bytes += bytes;
    size_t pk = g_dev_bytes_peak.load();
    while (now > pk && !g_dev_bytes_peak.compare_exchange_weak(pk, now)) {
    }
    return p;
}

// grow-only device buffer (capacity is kept across iterations and solves)
template <class T>
struct DevBuf {
    T *p = nullptr;
    size_t cap = 0;
    DevBuf() = default;
    DevBuf(const DevBuf &) = delete;
    DevBuf &operator=(const DevBuf &) = delete;
    DevBuf(DevBuf &&o) noexcept : p(o.p), cap(o.cap) { o.p = nullptr; o.cap = 0; }
    DevBuf &operator=(DevBuf &&o) noexcept {
        if (this != &o) { release(); p = o.p; cap = o.cap; o.p = nullptr; o.cap = 0; }
        return *this;
    }
    ~DevBuf() { release(); }
    void swap(DevBuf &o) noexcept { std::swap(p, o.p); std::swap(cap, o.cap); }
    // headroom for regrowth: a quarter, a sixteenth above 1 GiB
    static size_t with_headroom(size_t n) {
        if (n < 16) return 16;
        return n * sizeof(T) > (size_t(1) << 30) ? n + n / 16 : n + n / 4;
    }
    // contents are not kept
    T *ensure(size_t n) {
        if (n <= cap && p) return p;
        const size_t want = with_headroom(n);
        release();
        p = (T *)dev_alloc(want * sizeof(T));
        cap = want;
        return p;
    }
    // keeps the first `used` elements (copied on stream st); the old and the
    // new allocation coexist during the copy
    T *grow_keep(size_t n, size_t used, cudaStream_t st) {
        if (n <= cap && p) return p;
        const size_t want = with_headroom(n);
        T *q = (T *)dev_alloc(want * sizeof(T));
        if (p && used) {
            cudaError_t e = cudaMemcpyAsync(q, p, used * sizeof(T), cudaMemcpyDeviceToDevice, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) {
                cudaFree(q);
                g_dev_bytes -= want * sizeof(T);
                throw Error{-4, std::string("buffer regrowth copy: ") + cudaGetErrorString(e)};
            }
        }
        release();
        p = q;
        cap = want;
        return p;
    }
    void release() {
        if (p) {
            cudaFree(p);
            g_dev_bytes -= cap * sizeof(T);
        }
        p = nullptr;
        cap = 0;
    }
};

// per-system scalars kept on the device (FP64 where the method needs it)
struct SysDev {
    DevBuf<int> row0, nbs, n_orb;      // [S]
    DevBuf<int> sys_of_row;            // [NB]
    DevBuf<double> emin, emax;         // [S]
    // scalars of the current step, one buffer that a step uploads in one copy
    template <class T>
    struct View { T *p = nullptr; };
    DevBuf<double> step;               // c_lin, c_sq, tau0, tau1 [S], then active, tier [S] (int)
    View<double> c_lin, c_sq;          // branch coefficients
    View<double> tau0, tau1;           // truncation thresholds
    View<int> active;                  // 1 = still iterating
    View<int> tier;
    static size_t step_doubles(int S) { return (size_t)5 * S; }
    void ensure_step(int S) {
        double *q = step.ensure(step_doubles(S));
        c_lin.p = q; c_sq.p = q + S; tau0.p = q + 2 * (size_t)S; tau1.p = q + 3 * (size_t)S;
        active.p = reinterpret_cast<int *>(q + 4 * (size_t)S); tier.p = active.p + S;
    }
};

struct MatSet {
    int nmat = 0;
    int NB = 0;
    int b = 0;
    DevBuf<int> row_ptr;      // nmat*NB+1 (flat)
    DevBuf<int> col;          // total blocks
    DevBuf<double> val;       // total*b*b
    DevBuf<float> nrm;        // total
    DevBuf<uint16_t> ophi;    // tensor-core operand planes (hi and lo interleaved, 4 KB per block)
    DevBuf<float> opf32;      // FP32 operand copy for the CUDA-core FP32 products (hi word)
    DevBuf<float> opf32lo;    // lo word (x - hi) for the double-FP32 products
    std::vector<int64_t> nnzb;   // host copy, per matrix
    int64_t total = 0;
    // arithmetic (Arith) whose operand planes ophi holds for these values, with
    // the transposed positions, scales and FP32 copy in TcWork as of
    // TcWork::gen == planes_gen; -1: none
    int planes_ar = -1;
    uint64_t planes_gen = 0;
    void release() {
        planes_ar = -1;
        row_ptr.release(); col.release(); val.release(); nrm.release();
        ophi.release(); opf32.release(); opf32lo.release();
        nnzb.clear(); total = 0;
    }
};

// One output matrix of a multiplication step:
//   C = c_lin * X + c_sq * sum_t (A_t B_t)
struct Job {
    int out;          // output matrix index
    int xmat;         // matrix of the linear term (-1: none)
    int nterm;        // 1 or 2
    int a[2], b[2];   // operand matrices of each term
    int tau_sel;      // 0: tau0[s], 1: tau1[s]
};

constexpr int kMaxJobs = 8;
struct JobTable {
    int njob;
    Job job[kMaxJobs];
};

// Operand arithmetic of a numeric launch
// (AR_FF: double-FP32 products on the FP32 pipe, about 46 bits; AR_OZ:
// exact bf16 slice products on the tensor cores, 7 slices, FP64-class; AR_OZ8:
// FP64 products as 8-slice products)
enum Arith { AR_FP64 = 0, AR_FP32 = 1, AR_BF16X3 = 2, AR_FP16X3 = 3, AR_FF = 5, AR_OZ = 6, AR_OZ8 = 7 };

// Jobs selected per precision tier: bit p of m[t] selects job p for the rows
// of systems currently in tier t (systems of a batch move through the tiers
// independently)
constexpr int kMaxTiers = 4;
struct JobMask {
    unsigned m[kMaxTiers];
};

// ---------------------------------------------------------------------------
// kernel launchers (implemented in the k_*.cu files)
// ---------------------------------------------------------------------------

// k_scan.cu: exclusive scan (out may alias in); returns nothing, total at out[n].
void scan_exclusive_i64(const int *in, int64_t *out, int n, int64_t *tmp, cudaStream_t st);
// two counts per element (low and high 32 bits), totals below 2^31 each
void scan_exclusive_pair(const int64_t *in, int *out_lo, int *out_hi, int n, int64_t *tmp, cudaStream_t st);
size_t scan_tmp_elems(int n);

// k_setup.cu
void launch_gershgorin(const int *row_ptr, const int *col, const double *val, int NB, int b,
                       const int *sys_of_row, const int *row0, const int *n_orb,
                       double *row_lo, double *row_hi, cudaStream_t st);
void launch_sys_minmax(const double *row_lo, const double *row_hi, const int *row0, const int *nbs,
                       int S, double *emin, double *emax, cudaStream_t st);
// X := alpha * (diag_shift_sel ? emax[s] I : 0) + beta * H   (per system scaling), norms
// rows = number of block rows of the (possibly multi-matrix) set; NB = rows per matrix
void launch_init_scale(const int *row_ptr, const int *col, const double *hval, double *xval,
                       float *xnrm, int rows, int NB, int b, const int *sys_of_row,
                       const int *row0, const int *n_orb, const double *emin,
                       const double *emax, int is_x0, cudaStream_t st);
void launch_block_norms(const double *val, float *nrm, int64_t nblk, int b, cudaStream_t st);
// norm bounds equal for every block and its mirror (the larger of the two)
void launch_symmetric_norms(const int *row_ptr, const int *col, float *nrm, int nmat, int NB, cudaStream_t st);
void launch_check_values(const int *row_ptr, const int *col, const double *val, int64_t nval,
                         int NB, int b, const int *sys_of_row, const int *row0, const int *n_orb,
                         double rel_tol, int *err, cudaStream_t st);

// k_stats.cu: per-row partial sums then a deterministic per-system reduction.
// q-layout of the per-system output (double, [S][nq]):
//   0: Tr X0, 1: ||X0||_F^2, 2: Tr(X0 H0), 3+g: Tr(X1_g H0)
// A block row's sums come in row_stats_parts() partial sums: row_part has
// [q][NB][parts] entries.
int row_stats_parts();
void launch_row_stats(const int *row_ptr, const int *col, const double *val, int nmat, int NB,
                      int b, const int *h_row_ptr, const int *h_col, const double *h_val,
                      double *row_part, cudaStream_t st);
// Tr X and ||X||_F^2 of one matrix, row_part [2][NB]
void launch_row_trace_norm(const int *row_ptr, const int *col, const double *val, int NB, int b, double *row_part,
                           cudaStream_t st);
void launch_sys_sum(const double *row_part, int nq, int NB, const int *row0, const int *nbs,
                    int S, double *out, cudaStream_t st, int parts = 1);

// alpha: per-row partials of <P1_d, H1_g> over intersecting blocks
void launch_row_dots(const int *p_row_ptr, const int *p_col, const double *p_val, int np,
                     const int *h_row_ptr, const int *h_col, const double *h_val, int nh,
                     int NB, int b, double *row_part, cudaStream_t st);

// k_symbolic.cu
struct SymOut {
    int64_t *row_cnt;    // [njob*NB] kept blocks per (job,row); high 32 bits: those with col >= row
    int *row_off;        // [njob*NB] offset of the row's list in the pool
    int *pool_col;       // pool of kept columns
    int *pool_npair;     // pool of pair counts (per kept column)
    int *pool_top;       // [1] pool allocation counter
    int pool_cap;
    int *overflow;       // [1] set when the pool is too small
    unsigned long long *npairs;   // [njob] pairs of the kept upper-triangle blocks
};
// largest system (in block rows) the shared-memory row accumulator handles
constexpr int kSymMaxNs = 8192;
void launch_symbolic(const MatSet &in, const JobTable &jt, const SysDev &sd, int S,
                     SymOut so, cudaStream_t st, int max_ns);
// Gathers the pool into the output pattern: columns, row and job of every
// slot, its pair count (slot_npair may be null), and uidx, the rank of an
// upper slot (col >= row) among the upper slots (out_urp: their count before
// each row); slot_t of a lower slot is -1 until launch_pairs finds its partner.
// cls accumulates the pairs of active systems per kernel class.
constexpr int kClasses = 6;
struct ClassMasks {
    JobMask m[kClasses]; // tensor cores, FP64 FMAs, FP32, double-FP32, 7 slices, 8 slices (FP64 products)
};
void launch_gather(const SymOut &so, int njob, int NB, const int *out_row_ptr, const int *out_urp, int *out_col,
                   int *slot_row, int *slot_job, int *slot_npair, int *uidx, int *slot_t, const SysDev &sd,
                   const ClassMasks &cm, unsigned long long *cls, cudaStream_t st);
// pair lists of the jobs in `fill` (pair_off: offsets of every slot's list;
// null when no job is) and slot_x / slot_t of every slot
void launch_pairs(const MatSet &in, const JobTable &jt, const SysDev &sd, const int *out_row_ptr,
                  const int *out_col, const int *slot_row, const int *slot_job,
                  const int64_t *pair_off, int64_t nslot, int NB, int *pair_a, int *pair_b,
                  int *slot_x, int *slot_t, int *err, cudaStream_t st, JobMask fill);

// A product kernel that computes in FP32 leaves its untruncated block in FP32
// (kBlockF32 in the slot's keep byte) and the compaction widens it: element
// (r, c) of the b x b block at this index of the slot.  Four columns of a row
// are adjacent and the rows follow, so that a lane that holds a row writes 16
// bytes beside its neighbours', and the compaction reads the block's rows and
// its columns (for the transposed block) equally well.  The FP32 copies of
// the old blocks for the linear terms have the same layout.
constexpr uint8_t kKeepBlock = 1, kBlockF32 = 2;
__host__ __device__ inline int f32_index(int b, int r, int c) { return ((c >> 2) * b + r) * 4 + (c & 3); }

// k_numeric.cu: C(upper slot) = c_lin X + c_sq sum(pairs); lower slot = transpose
struct NumArgs {
    const double *in_val;
    const float *in_f32;       // FP32 copy of in_val (FP32 products), may be null
    const int *tpos;           // position of every block's transpose (with in_f32 and b = 32)
    const float *in_f32lo;     // in_val - in_f32 rounded to FP32 (double-FP32 products), may be null
    const int *pair_a, *pair_b;
    const int64_t *pair_off;   // null: no slot has pairs (copies of converged systems only)
    const int *slot_row, *slot_job, *slot_x, *slot_t;
    const int *work;        // upper slots to process
    const int *nwork;       // their number
    int *work_next;         // zeroed counter: next work item to hand out
    int max_work;           // bound of *nwork
    const int *sys_of_row;
    const double *c_lin, *c_sq, *tau0, *tau1;
    const int *active;
    int job_tau_sel[kMaxJobs];
    // outputs: only upper-triangle slots (col >= row) are computed; the
    // values of upper slot s go to out_val at index uidx[s] - u0 (uidx: rank
    // of s among the upper slots, u0: that of the group's first one);
    // (b*b doubles apart; FP64, or FP32 as kBlockF32 says), norm bound and
    // keep flag to out_nrm[s], keep[s]
    double *out_val;
    float *out_nrm;
    uint8_t *keep;
    const int *uidx;
    int64_t u0;
    int b;
};
void launch_numeric_simt(const NumArgs &a, Arith ar, cudaStream_t st);
// diagonal elements of the one-term products A A of the jobs in `jobs` as FP64
// FMA chains, over those in out_val; flat rows [r0, r0 + nrows) of the mask
void launch_diag_fp64(const NumArgs &a, const MatSet &in, const JobTable &jt, JobMask jobs, const int *out_rp,
                      const int *out_col, const int *sys_tier, int r0, int nrows, cudaStream_t st);
// FP32 copy of the FP64 master values (for the FP32 products)
// FP32 copy (and, with f32lo, the FP32 remainder) of FP64 values
void launch_to_f32(const double *val, float *f32, int64_t n, cudaStream_t st, float *f32lo = nullptr);

// k_compact.cu
// upper slots of the active systems' jobs selected by job_mask (per system
// tier), plus (with_inactive) all upper slots of converged systems
// (slots [s0, s1) only)
void launch_build_work(const int *slot_row, const int *out_col, int64_t s0, int64_t s1,
                       int *work, int *nwork, cudaStream_t st, const int *sys_of_row,
                       const int *active, const int *slot_job, const int *sys_tier, JobMask job_mask,
                       int with_inactive);
// Compaction of the rows [r0, r0 + nrows) of the mask.  An upper slot is kept
// on its own flag; a lower slot t on that of its upper partner slot_t[t],
// (a slot without a partner is dropped, whatever its flag: no index is taken
// from it, and the host reads the error bit of the pair lists afterwards)
// and receives that block's transpose, read from out_val when the partner
// belongs to the current group (uidx >= u0) and otherwise from the already
// compacted output (dest[partner]).  dest[s] receives the output position of
// every kept upper slot s.
struct CompactArgs {
    const int *out_rp, *out_col, *slot_row, *slot_t, *uidx;
    const double *out_val;
    const float *out_nrm;
    const uint8_t *keep;
    int64_t u0;
    int *dest;
    int *src;               // [kept blocks of the group]: slot of output block d0 + k
    int *new_rp, *new_col;
    double *new_val;
    float *new_nrm;
    int r0, nrows, b;
    int d0;                 // first output block of the group
    int NB;
    unsigned *mx;           // per matrix: largest block norm of the group (bit pattern)
    unsigned long long *look;
    int look_polls;         // bound of the waits for other CTAs (lookback.cuh)
    int *look_err;          // set when one ran out: the pattern is not complete and no values are copied
    // the next step's operands (null: not made): planes at the transposed
    // positions, those positions, operand scales, FP32 copy for the linear
    // terms (may be null)
    uint16_t *planes;
    int *tpos;
    float *scale, *xlin;
    int bf16, njob;
    const int *slot_job;
};
// pattern of the kept blocks of rows [r0, r0 + nrows) (`look`:
// compact_look_words(nrows) zeroed words, for mx and look), then the values of its
// kept blocks (at most max_blocks; how many is read on the device).  In a pattern
// that a wait cut short, row pointers and columns lie inside the mask's room.
int64_t compact_look_words(int nrows);
void launch_compact_rows(CompactArgs &c, unsigned long long *look, cudaStream_t st);

// device counters of a multiplication step (ints)
enum {
    kCtrTop = 0,         // pool_top, overflow of the symbolic phase
    kCtrErr = 2,         // error bits of the pair lists
    kCtrPairs = 4,       // 64 bits per job: pairs of its upper slots
    kCtrClass = kCtrPairs + 2 * kMaxJobs,   // kClasses x 64 bits: pairs per kernel class
    kCtrWork = 32,       // work items of the three CUDA-core classes (zeroed for every group, with the next)
    kCtrNext = 36,       // next item to hand out, per class
    kCtrLook = 39,       // a wait of the compaction ran out
    kCtrInts = 40        // even: 64-bit words follow
};
static_assert(kCtrClass + 2 * kClasses <= kCtrWork && kCtrInts % 2 == 0, "counters");
// what the host reads of a step, in page-locked memory
struct HostStep {
    int ctr[kCtrInts];
    int kept;
    int upper[kMaxJobs + 1];          // upper slots before every job, and their number
    int tc[8], oz[8];                 // TcWork::counters of the two plans
    int pre_err;                      // error bits of the transposed positions (FP32 products)
    int rp[kMaxJobs + 1];             // first block of every output matrix
};
// one launch that writes the listed values (null: not this one) into *dst,
// which the host reads after its next wait; upper, rp: every NB-th entry of the
// upper slots' and of the result's row pointers
struct PublishArgs {
    HostStep *dst;
    const int *ctr, *upper, *kept, *tc, *oz, *pre_err, *rp;
    int NB, njob;
};
void launch_publish(const PublishArgs &a, cudaStream_t st);
void launch_compact_copy(const CompactArgs &c, int max_blocks, cudaStream_t st);

// k_lowdin.cu: out = fac[sys] * val for every block of the first NB block rows
// (pad_one: the diagonal of padding rows set to 1), and identity blocks.
void launch_scale_sys(const int *row_ptr, const int *col, const double *val, int NB, int b, const int *sys_of_row,
                      const int *row0, const int *n_orb, const double *fac, int pad_one, double *out,
                      cudaStream_t st);
void launch_identity_blocks(double *val, int64_t nblk, int b, cudaStream_t st);

// k_reblock.cu: the same matrix in b_out x b_out instead of b_in x b_in blocks.
// Host pattern (rp/col of one matrix, local block indices; n orbitals): an
// output block exists where a stored input block overlaps it.
void reblock_pattern(const std::vector<int> &rp, const std::vector<int> &col, int b_in, int n, int b_out,
                     std::vector<int> &rp_out, std::vector<int> &col_out);
// Values of the nout output blocks (out_row/out_col: block row and column of
// each, device) from the input matrix (device row_ptr/col/val, nb_in rows).
void launch_reblock_vals(const int *in_rp, const int *in_col, const double *in_val, int nb_in, int b_in,
                         const int *out_row, const int *out_col, double *out_val, int64_t nout, int b_out,
                         cudaStream_t st);

}  // namespace rdm

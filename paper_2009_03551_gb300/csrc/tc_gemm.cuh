// Tensor-core (tcgen05) numeric phase: declarations shared with the driver.
#pragma once

#include "rdm_internal.cuh"

namespace rdm {

// Test settings of the tensor-core path (rdm_set_test_knobs); zeros keep the
// production behaviour.
constexpr int kInjectTileWait = 1, kInjectRowWait = 2, kInjectStepRoom = 4;
struct TcKnobs {
    int inject = 0;             // kInject*: failures of one plan or compaction to come
    int fail_alloc = 0;         // > 0: that many device allocations of the steps on, one fails
    long long wait_cycles = 0;  // bound of every mbarrier wait in SM clock cycles (0: ~2 s)
    int hold = 0;               // 1: the MMA thread first waits for a flag that nothing sets
    int window_words = 0;       // bitmap window of the tile-plan builders in 32-column words
                                // (0: 512, i.e. 16,384 columns; wider windows take the serial merge)
    int block_copies = 0;       // 1: planes at their own positions and one bulk copy per block
};

// work buffers of the tensor-core path (tile lists, per-tile K-step lists)
struct TcWork {
    TcKnobs knobs;
    DevBuf<uint16_t> zero;      // zero operand blocks: one per CTA and K-step slot
    DevBuf<int> tiles;          // per tile: job, I, -, nsteps, mask slot[TBM x TBN], column j[TBN]
    DevBuf<int64_t> step_rng;   // per tile: its K-steps are [step_rng[2 t], step_rng[2 t + 1])
    int64_t need_steps = 0;     // K-steps of a plan that did not fit (0: fits)
    DevBuf<int> steps;          // per K-step: TBM A block indices, TBN B block indices (-1 = zero)
    // [0]: error bits of the product kernel, [1]: a list outgrew its buffer
    // (the product kernel then does nothing), [2]: tiles, [3]: the tile list is not
    // complete (a wait ran out; the lists are built again), [4..5]: K-steps (64
    // bits), [6]: tiles handed out, [8..]: state of the tile list's prefix sums.  plan_counter_ints(units)
    // ints of the caller's memory, zeroed before a plan is built
    int *counters = nullptr;
    DevBuf<float> scale;        // per matrix: power-of-two scale of its operand planes
    DevBuf<int> tpos;           // per block (i, k) of the input set: global index of block (k, i)
    // [0]: error bits of the operand preparation (8: a transposed block missing);
    // [1 + m]: largest block norm of matrix m (bit pattern)
    DevBuf<int> pre_err;
    DevBuf<float> xlin;         // FP32 values of the input set's upper blocks (layout f32_index)
    bool lin = false;           // xlin is filled for this step
    uint64_t gen = 0;           // counts the rewrites of tpos, scale and xlin
    bool lean = false;          // memory is short: no FP32 copy
    bool xlin_valid = false;    // xlin was written with the planes
    bool tpos_valid = false;    // the planes sit at tpos and the K-step lists point there
};

// work buffers of the slice-product (FP64-class) tensor-core path
struct OzWork {
    int nslice = 0;             // bf16 slices per element: 7 or 8
    DevBuf<int> e;              // per flat row: exponent e_r of its scale 2^e_r
    DevBuf<int> row_of;         // flat block row of every block
    DevBuf<uint16_t> slices_a, slices_b;   // the slices of every block as A and as B operand (2 KB per slice)
    DevBuf<uint16_t> zero;      // zero blocks: one per CTA and K-step slot
};

// Lists of one launch.  Their lengths stay on the device (TcWork::counters);
// the host has bounds.
struct TcPlan {
    int max_tile = 0;           // bound of the number of tiles (0: no tile)
    int64_t cap_steps = 0;      // K-steps that the list has room for
};

// Block sizes the tensor-core kernel handles (16, 32, 64), and the block rows
// of its 128 x 256 tiles for block size b (128 / b; 4 for other sizes, the
// super-row of the CUDA-core path).
bool tc_block_size_ok(int b);
int tc_tile_rows(int b);
int64_t plan_counter_ints(int units);

// Convert the FP64 master values of `in` into hi/lo operand planes of
// arithmetic `ar` in the K-major core-matrix layout of the MMA.  For fp16
// every matrix is first scaled by a power of two (from its largest block
// norm) so that its values sit in the normal range of fp16; the product
// kernel divides the scale back out per job.
void prepare_operands(MatSet &in, Arith ar, bool lin, TcWork &w, cudaStream_t st);

// The operands of `in` as the compaction left them (MatSet::planes_ar), if they
// are those of arithmetic `ar`; false: prepare_operands has to make them.
bool reuse_operands(const MatSet &in, Arith ar, bool lin, TcWork &w);
// Room for the operands of `out` (kept blocks, njob matrices) and their
// pointers in `c`, for the compaction to write; `planes`: the buffer of the input
// set's operands, which the step no longer reads.
void operands_from_compaction(CompactArgs &c, MatSet &out, DevBuf<uint16_t> &planes, int64_t kept, int njob, Arith ar,
                              TcWork &w);

// Positions of the transposed blocks of the set (w.tpos); a pattern that is not
// symmetric sets error bit 8 of pre_err[0].
void find_transposes(const MatSet &in, TcWork &w, cudaStream_t st);

// Tile and K-step lists of one multiplication step from the output mask, for
// the jobs selected by job_mask (per system tier) and the super-row units
// [unit0, unit1) (unit = job * ceil(NB/TR) + I covers block rows
// TR I .. TR I + TR - 1 of the job, TR = tc_tile_rows(b)); those of the selected
// jobs have nupper upper slots.  Nothing is waited for: min_steps is the least room made for
// K-steps, and a list that needs more (counters[1], with the number in
// counters[4..5]) has to be built again.
TcPlan build_tc_plan(const MatSet &in, const JobTable &jt, const SysDev &sd, const int *out_rp,
                     const int *mcol, TcWork &w, JobMask job_mask, int unit0, int unit1, int64_t nupper,
                     int64_t min_steps, cudaStream_t st);

// Numeric phase on the tensor cores; same output contract as
// launch_numeric_simt for the slots of active systems.
void launch_numeric_tc(const NumArgs &a, const MatSet &in, const JobTable &jt, Arith ar, TcWork &w,
                       const TcPlan &plan, cudaStream_t st);

// FP64-class products on the tensor cores from exact bf16 slices (32 x 32
// blocks; k_oz.cu): the slices (7 or 8 per element) and row scales of the
// first nmat matrices of `in` (false, with nothing done, when the device has
// no room for them; then the caller has another way), the tile lists (128 x 64 tiles) of the jobs in job_mask,
// and the launch (same output contract as the other numeric launches).
// tc_step_flops / oz_step_flops: the MMA flops issued per K-step; reserve:
// bytes the slices leave free.
bool prepare_oz_operands(const MatSet &in, int nmat, int slices, size_t reserve, OzWork &w, cudaStream_t st);
TcPlan build_oz_plan(const MatSet &in, const JobTable &jt, const SysDev &sd, const int *out_rp, const int *mcol,
                     TcWork &w, JobMask job_mask, int unit0, int unit1, int64_t nupper, int64_t min_steps,
                     cudaStream_t st);
double tc_step_flops(int b);
double oz_step_flops(const OzWork &ow);
void launch_numeric_oz(const NumArgs &a, const MatSet &in, const JobTable &jt, const int *mcol, OzWork &ow,
                         TcWork &w, const TcPlan &plan, cudaStream_t st);

}  // namespace rdm

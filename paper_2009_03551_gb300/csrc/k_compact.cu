// Stream compaction after truncation: the pattern and norm bounds of the kept
// blocks, with the new row pointers, and an order-preserving copy of their
// values; the products compute only
// the upper triangle and the copy writes each lower block as the transpose
// of its upper partner.  Also builds the work list of upper-triangle output
// blocks for the numeric phase.
#include "fp_bits.cuh"
#include "lookback.cuh"
#include "rdm_internal.cuh"
#include "tc_split.cuh"

#include <algorithm>

namespace rdm {
namespace {

// work list: slots with col >= row, in slot order (one warp per 32 slots,
// ballot-ordered, block-level offsets through one atomic per warp; the order
// of the list does not affect results)
// keeps the upper slots of the active systems' jobs in job_mask and, with
// with_inactive, every upper slot of a converged system (those are copied)
__global__ void k_build_work(const int *__restrict__ slot_row, const int *__restrict__ out_col,
                             int64_t s0, int64_t s1, int *work, int *nwork, const int *__restrict__ sys_of_row,
                             const int *__restrict__ active, const int *__restrict__ slot_job,
                             const int *__restrict__ sys_tier, JobMask job_mask, int with_inactive) {
    int64_t s = s0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int lane = threadIdx.x & 31;
    bool up = s < s1 && out_col[s] >= slot_row[s];
    if (up) {
        const int sys = sys_of_row[slot_row[s]];
        const bool act = active[sys] != 0;
        up = act ? ((job_mask.m[sys_tier[sys] & (kMaxTiers - 1)] >> slot_job[s]) & 1u) != 0 : with_inactive != 0;
    }
    unsigned m = __ballot_sync(0xffffffffu, up);
    int base = 0;
    if (lane == 0 && m) base = atomicAdd(nwork, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (up) work[base + __popc(m & ((1u << lane) - 1u))] = (int)s;
}

// One warp per row of the group: the kept blocks (an upper slot on its own flag,
// a lower one on its upper partner's) are counted, the row gets its place from
// the running sums of the CTAs before it, and their columns, norm bounds and
// destinations are written in order; src[d - d0] receives the slot of output
// block d, mx[m] the largest norm of matrix m.  Bound by launches and waits for
// loads: one launch where count, scan and copy were three (150-atom cluster:
// 16 us, 9 us so).
constexpr int kRowWarps = 8;
__global__ void __launch_bounds__(32 * kRowWarps) k_compact_rows(CompactArgs c) {
    __shared__ int cnt_s[kRowWarps];
    __shared__ int sh_bid, sh_base;
    const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
    const int bid = lookback_id(c.look, &sh_bid);
    const int r = c.r0 + bid * kRowWarps + wq;
    const bool row = r < c.r0 + c.nrows;
    const int rbeg = row ? c.out_rp[r] : 0, rend = row ? c.out_rp[r + 1] : 0;
    int n = 0;
    for (int p = rbeg + lane; p < rend; p += 32) {
        const int partner = c.slot_t[p];     // -1: the mask lacks it
        n += partner >= 0 ? c.keep[c.out_col[p] >= c.slot_row[p] ? p : partner] & kKeepBlock : 0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if (lane == 0) cnt_s[wq] = n;
    __syncthreads();
    int total = 0, before = 0;
#pragma unroll
    for (int k = 0; k < kRowWarps; ++k) {
        if (k < wq) before += cnt_s[k];
        total += cnt_s[k];
    }
    if (wq == 0) {
        const int first = lookback_sum(c.look, bid, total, c.look_err, c.look_polls) + c.d0;
        if (lane == 0) {
            sh_base = first;
            if (bid == (int)gridDim.x - 1) c.new_rp[c.r0 + c.nrows] = first + total;
        }
    }
    __syncthreads();
    int dst = sh_base + before;
    if (row && lane == 0) c.new_rp[r] = dst;
    float mx = 0.f;
    for (int base = rbeg; base < rend; base += 32) {
        const int p = base + lane;
        bool k = false;
        int src = p;
        if (p < rend) {
            const int partner = c.slot_t[p];
            src = c.out_col[p] >= c.slot_row[p] ? p : partner;
            k = partner >= 0 && (c.keep[src] & kKeepBlock);
        }
        const unsigned m = __ballot_sync(0xffffffffu, k);
        if (k) {
            const int d = dst + __popc(m & ((1u << lane) - 1u));
            c.new_col[d] = c.out_col[p];
            const float nrm = c.out_nrm[src];
            c.new_nrm[d] = nrm;
            mx = fmaxf(mx, nrm);
            c.src[d - c.d0] = p;
            c.dest[p] = d;
        }
        dst += __popc(m);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (row && lane == 0 && mx > 0.f) atomicMax(&c.mx[r / c.NB], __float_as_uint(mx));
}

// A step's counters and sizes to page-locked host memory, in one launch: a copy
// each holds the stream up for ~2 us, and a step had seven of them.
constexpr int kPublishThreads = 64;    // a thread per counter: one load's latency
__global__ void __launch_bounds__(kPublishThreads) k_publish(PublishArgs a) {
    static_assert(kCtrInts <= kPublishThreads && kMaxJobs < kPublishThreads, "one thread per value");
    const int t = threadIdx.x;
    if (a.ctr && t < kCtrInts) a.dst->ctr[t] = a.ctr[t];
    if (a.tc && t < 8) a.dst->tc[t] = a.tc[t];
    if (a.oz && t < 8) a.dst->oz[t] = a.oz[t];
    if (a.rp && t <= a.njob) a.dst->rp[t] = a.rp[(size_t)t * a.NB];
    if (a.upper && t <= a.njob) a.dst->upper[t] = a.upper[(size_t)t * a.NB];
    if (t == 0) {
        if (a.kept) a.dst->kept = *a.kept;
        if (a.pre_err) a.dst->pre_err = *a.pre_err;
    }
}

// Values of the kept blocks, block sizes that the tensor cores do not take: one
// CTA per block (grid-stride), upper blocks are copied, lower ones transposed
// through shared memory (b x (b+1) doubles) from their upper partner, which is
// in this group's buffer or already compacted.
__global__ void __launch_bounds__(128) k_compact_vals(CompactArgs c) {
    extern __shared__ double tile[];
    // nothing where src is not complete: the host repeats the step
    const int bad = *c.look_err, end = c.new_rp[c.r0 + c.nrows], d1 = bad ? c.d0 : end;
    const int b = c.b, bb = b * b, ld = b + 1;
    for (int d = c.d0 + blockIdx.x; d < d1; d += gridDim.x) {
        const int p = c.src[d - c.d0];
        double *out = c.new_val + (size_t)d * bb;
        if (c.out_col[p] >= c.slot_row[p]) {
            const double *s = c.out_val + (size_t)(c.uidx[p] - c.u0) * bb;
            for (int e = threadIdx.x; e < bb; e += blockDim.x) out[e] = s[e];
        } else {
            const int t = c.slot_t[p];
            const int ut = c.uidx[t];
            const double *s = ut >= c.u0 ? c.out_val + (size_t)(ut - c.u0) * bb
                                         : c.new_val + (size_t)c.dest[t] * bb;
            for (int e = threadIdx.x; e < bb; e += blockDim.x) tile[(e / b) * ld + (e % b)] = s[e];
            __syncthreads();
            for (int e = threadIdx.x; e < bb; e += blockDim.x) out[e] = tile[(e % b) * ld + (e / b)];
            __syncthreads();
        }
    }
}

// The same for B = 16, 32, 64, a warp per block, without shared memory: a lane
// takes 8 neighbouring columns of a row of an upper block, and for a lower
// block 8 rows x 4 columns of its partner, which are 8 neighbouring columns of
// 4 rows of the transpose.  FP32 sources (kBlockF32) are widened.  PL = 1 (fp16)
// or 2 (bf16): the same pass writes the next step's operand planes, at the
// transposed block's position, and the FP32 copy for its linear terms, instead
// of a second one that reads the FP64 values back.  Bound by memory: 18 bytes
// per element of the result where the two passes moved 26 (2,000-atom cluster,
// 300,000 blocks of 32: 292 + 271 us per step in two passes, 537 in one;
// 150 atoms, 5,500 blocks: 16.5 + 13.5 us, 21 in one, and four launches less).
template <int B, int PL>
__global__ void __launch_bounds__(128) k_compact_blocks(CompactArgs c) {
    const int bad = *c.look_err, end = c.new_rp[c.r0 + c.nrows], d1 = bad ? c.d0 : end;
    constexpr int BB = B * B, C8 = B / 8;
    const int lane = threadIdx.x & 31;
    if (PL && blockIdx.x == 0 && (int)threadIdx.x < c.njob) c.scale[threadIdx.x] = matrix_scale(c.mx[threadIdx.x], PL == 1);
    for (int d = c.d0 + blockIdx.x * 4 + (threadIdx.x >> 5); d < d1; d += gridDim.x * 4) {
        const int p = c.src[d - c.d0];
        double *out = c.new_val + (size_t)d * BB;
        const bool up = c.out_col[p] >= c.slot_row[p];
        const int partner = c.slot_t[p], t = up ? p : partner;
        const int ut = c.uidx[t];
        const bool here = ut >= c.u0;
        const double *s = here ? c.out_val + (size_t)(ut - c.u0) * BB : c.new_val + (size_t)c.dest[t] * BB;
        const float4 *f = here && (c.keep[t] & kBlockF32) ? reinterpret_cast<const float4 *>(s) : nullptr;
        uint16_t *planes = nullptr;
        float sc = 1.f;
        if constexpr (PL != 0) {
            const int at = c.dest[partner];
            if (lane == 0) c.tpos[d] = at;
            planes = c.planes + (size_t)at * (2 * BB);
            sc = matrix_scale(c.mx[c.slot_job[p]], PL == 1);
        }
        if (up) {
            for (int k = lane; k < B * C8; k += 32) {
                const int r = k / C8, c0 = 8 * (k % C8);
                double v[2][4];
                float x[8];
                if (f) {
                    const float4 a0 = f[(c0 >> 2) * B + r], a1 = f[((c0 >> 2) + 1) * B + r];
                    x[0] = a0.x; x[1] = a0.y; x[2] = a0.z; x[3] = a0.w;
                    x[4] = a1.x; x[5] = a1.y; x[6] = a1.z; x[7] = a1.w;
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u >> 2][u & 3] = f32_to_f64(x[u]);
                } else {
                    ld_f64x4(s + r * B + c0, v[0]);
                    ld_f64x4(s + r * B + c0 + 4, v[1]);
                    if constexpr (PL != 0) {
#pragma unroll
                        for (int u = 0; u < 8; ++u) x[u] = f64_to_f32(v[u >> 2][u & 3]);
                    }
                }
                st_f64x4(out + r * B + c0, v[0]);
                st_f64x4(out + r * B + c0 + 4, v[1]);
                if constexpr (PL != 0) {
                    store_planes<PL == 2, B>(planes, r, c0, x, sc);
                    if (c.xlin) {
                        float *xl = c.xlin + (size_t)d * BB;
                        *reinterpret_cast<float4 *>(xl + f32_index(B, r, c0)) = make_float4(x[0], x[1], x[2], x[3]);
                        *reinterpret_cast<float4 *>(xl + f32_index(B, r, c0 + 4)) = make_float4(x[4], x[5], x[6], x[7]);
                    }
                }
            }
        } else {
            for (int k = lane; k < (B / 4) * C8; k += 32) {
                const int c4 = k / C8, r0 = 8 * (k % C8);       // source columns 4 c4 .., rows r0 ..
                if (f) {
                    float4 a[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) a[q] = f[c4 * B + r0 + q];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        float x[8];
                        double v[2][4];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            x[q] = u == 0 ? a[q].x : u == 1 ? a[q].y : u == 2 ? a[q].z : a[q].w;
                            v[q >> 2][q & 3] = f32_to_f64(x[q]);
                        }
                        st_f64x4(out + (4 * c4 + u) * B + r0, v[0]);
                        st_f64x4(out + (4 * c4 + u) * B + r0 + 4, v[1]);
                        if constexpr (PL != 0) store_planes<PL == 2, B>(planes, 4 * c4 + u, r0, x, sc);
                    }
                } else {
                    double a[8][4];
#pragma unroll
                    for (int q = 0; q < 8; ++q) ld_f64x4(s + (r0 + q) * B + 4 * c4, a[q]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        double v[2][4];
#pragma unroll
                        for (int q = 0; q < 8; ++q) v[q >> 2][q & 3] = a[q][u];
                        st_f64x4(out + (4 * c4 + u) * B + r0, v[0]);
                        st_f64x4(out + (4 * c4 + u) * B + r0 + 4, v[1]);
                        if constexpr (PL != 0) {
                            float x[8];
#pragma unroll
                            for (int q = 0; q < 8; ++q) x[q] = f64_to_f32(a[q][u]);
                            store_planes<PL == 2, B>(planes, 4 * c4 + u, r0, x, sc);
                        }
                    }
                }
            }
        }
    }
}

template <int B>
void launch_blocks(const CompactArgs &c, int max_blocks, cudaStream_t st) {
    const int grid = (int)std::min((max_blocks + 3) / 4, 152 * 16);
    if (!c.planes) k_compact_blocks<B, 0><<<grid, 128, 0, st>>>(c);
    else if (c.bf16) k_compact_blocks<B, 2><<<grid, 128, 0, st>>>(c);
    else k_compact_blocks<B, 1><<<grid, 128, 0, st>>>(c);
    RDM_LAUNCH_CHECK();
}

}  // namespace

void launch_build_work(const int *slot_row, const int *out_col, int64_t s0, int64_t s1, int *work,
                       int *nwork, cudaStream_t st, const int *sys_of_row, const int *active,
                       const int *slot_job, const int *sys_tier, JobMask job_mask, int with_inactive) {
    if (s1 <= s0) return;
    int64_t grid = (s1 - s0 + 255) / 256;
    k_build_work<<<(unsigned)grid, 256, 0, st>>>(slot_row, out_col, s0, s1, work, nwork, sys_of_row,
                                                 active, slot_job, sys_tier, job_mask, with_inactive);
    RDM_LAUNCH_CHECK();
}

int64_t compact_look_words(int nrows) { return kMaxJobs + lookback_words((nrows + kRowWarps - 1) / kRowWarps); }

void launch_compact_rows(CompactArgs &c, unsigned long long *look, cudaStream_t st) {
    c.mx = reinterpret_cast<unsigned *>(look);
    c.look = look + kMaxJobs;
    if (c.nrows == 0) {
        RDM_CUDA_TRY(cudaMemsetAsync(const_cast<int *>(c.new_rp) + c.r0, 0, sizeof(int), st));
        return;
    }
    k_compact_rows<<<(c.nrows + kRowWarps - 1) / kRowWarps, kRowWarps * 32, 0, st>>>(c);
    RDM_LAUNCH_CHECK();
}

void launch_publish(const PublishArgs &a, cudaStream_t st) {
    k_publish<<<1, kPublishThreads, 0, st>>>(a);
    RDM_LAUNCH_CHECK();
}

void launch_compact_copy(const CompactArgs &c, int max_blocks, cudaStream_t st) {
    if (max_blocks <= 0 || c.nrows == 0) return;
    switch (c.b) {
        case 16: return launch_blocks<16>(c, max_blocks, st);
        case 32: return launch_blocks<32>(c, max_blocks, st);
        case 64: return launch_blocks<64>(c, max_blocks, st);
        default: break;
    }
    const size_t smem = (size_t)c.b * (c.b + 1) * sizeof(double);
    const int grid = std::min(max_blocks, 152 * 16);
    k_compact_vals<<<grid, 128, smem, st>>>(c);
    RDM_LAUNCH_CHECK();
}

}  // namespace rdm

// Tile and K-step lists of the tensor-core products (the symbolic half of
// Algorithm 1's Gustavson merge, lifted to tiles of TBM x TBN blocks), shared
// by the tensor-core kernels.  A geometry G supplies TBM, TBN, kSlots =
// TBM + TBN, kColOff = 4 + TBM * TBN and kTileInts = kColOff + TBN.
#pragma once

#include <algorithm>

#include "lookback.cuh"
#include "tc_gemm.cuh"

namespace rdm {
namespace {

template <int TBM_, int TBN_>
struct PlanGeo {
    static constexpr int TBM = TBM_;                    // block rows per tile
    static constexpr int TBN = TBN_;                    // block columns per tile
    static constexpr int kSlots = TBM + TBN;            // operand blocks per K-step: A rows, then B rows
    static constexpr int kColOff = 4 + TBM * TBN;       // tile record: job, super-row, steps of term 0, nsteps,
    static constexpr int kTileInts = kColOff + TBN;     //   mask slot[TBM x TBN], column j of each tile column
    static_assert(kSlots <= 32, "one producer lane per slot");
};

// ---------------------------------------------------------------------------
// tile lists
// ---------------------------------------------------------------------------
struct TileBuild {
    const int *rp;       // input set row_ptr (flat)
    const int *col;
    int NB, NBT;         // block rows, super-rows (ceil(NB / TBM))
    JobTable jt;
    const int *out_rp;   // mask row_ptr (flat, njob*NB+1)
    const int *mcol;     // mask columns
    const int *sys_of_row, *active, *sys_tier;
    JobMask job_mask;    // jobs computed on the tensor cores, per tier
    int u0, u1;          // super-row units (job * NBT + I) of this plan
    unsigned long long *look;   // running sums of k_tile_rows' CTAs (lookback.cuh), zeroed
    int look_polls;             // bound of its waits
    int *tiles;          // [ntile * kTileInts]
    int64_t *step_rng;   // [2 ntile]: a tile's K-steps are [step_rng[2 t], step_rng[2 t + 1])
    int *steps;          // [nsteps * kSlots]
    int64_t cap_steps;   // room in steps
    int *flags;          // TcWork::counters
    int max_words;       // bitmap window in 32-column words (<= 512); wider windows: serial merge
    const int *tpos;     // K-step entries point at tpos[e] (the planes' position), or at e if null
};

// upper mask range [cur, end) of block row TBM I + m of job p, empty for rows
// whose system is converged or whose job is not computed on the tensor cores
template <class G>
__device__ __forceinline__ void tile_row_range(const TileBuild &T, int p, int I, int m, int &cur, int &end) {
    const int i = G::TBM * I + m;
    cur = end = 0;
    if (i >= T.NB) return;
    int lo = T.out_rp[p * T.NB + i], hi = T.out_rp[p * T.NB + i + 1];
    end = hi;
    // first column >= i (upper triangle)
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (T.mcol[mid] < i) lo = mid + 1; else hi = mid;
    }
    cur = lo;
    // converged systems keep their blocks through the copy path of the
    // numeric phase, and jobs on the CUDA cores have their own launch:
    // neither produces tiles
    const int sys = T.sys_of_row[i];
    if (!T.active[sys] || !((T.job_mask.m[T.sys_tier[sys] & (kMaxTiers - 1)] >> p) & 1u)) cur = end;
}

// Tiles of one (job, super-row), warp-parallel: the upper mask columns of
// the TBM block rows are marked in a shared-memory bitmap over their column
// window; the rank of a column among the distinct ones (prefix popcounts)
// gives its tile (rank / TBN) and tile column (rank % TBN).  Windows wider
// than the bitmap fall back to a serial merge by lane 0.  The last super-rows
// come first, so that X0's tiles, with one product where X1's have two, end the
// list (the product kernel hands the tiles out in order, and a short one at the
// end leaves less idle).  The tiles of a CTA's super-rows alternate, the first
// of each, the second of each and so on, so that those in work at a time share
// operands both ways (2,000-atom cluster: 58.7 -> 57.3 ms of products).  A CTA
// gets the number of tiles before its own from the running sums of the CTAs
// before it, so that one launch counts and writes
// (40 super-rows of a 150-atom cluster: 19 us for count, scan and fill in three
// launches, 10 us in one).
constexpr int kTileRowWarps = 8, kTileRowWords = 512;   // 16,384 columns per window
template <class G, class Place>
__device__ int tile_rows_serial(const TileBuild &T, int p, int I, const int *cur0, const int *end0, const Place &place,
                                bool fill);
template <class G>
__global__ void __launch_bounds__(32 * kTileRowWarps) k_tile_rows(TileBuild T) {
    __shared__ unsigned bits_s[kTileRowWarps][kTileRowWords];
    __shared__ int rank_s[kTileRowWarps][kTileRowWords];
    __shared__ int cnt_s[kTileRowWarps];
    __shared__ int sh_bid, sh_base;
    const int wq = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bid = lookback_id(T.look, &sh_bid);
    const int t = T.u1 - 1 - (bid * kTileRowWarps + wq);
    const int p = max(t, 0) / T.NBT, I = max(t, 0) % T.NBT;
    unsigned *bm = bits_s[wq];
    int *wr = rank_s[wq];
    int c0 = 0, e0 = 0;
    if (t >= T.u0 && lane < G::TBM) tile_row_range<G>(T, p, I, lane, c0, e0);
    int cur[G::TBM], end[G::TBM];
    int lo = 0x7fffffff, hi = -1;
#pragma unroll
    for (int m = 0; m < G::TBM; ++m) {
        cur[m] = __shfl_sync(0xffffffffu, c0, m);
        end[m] = __shfl_sync(0xffffffffu, e0, m);
        if (cur[m] < end[m]) {
            lo = min(lo, T.mcol[cur[m]]);
            hi = max(hi, T.mcol[end[m] - 1]);
        }
    }
    const int nw = hi < lo ? 0 : ((hi - lo) >> 5) + 1;
    const bool serial = nw > T.max_words;
    int ntile = 0;
    if (serial) {
        if (lane == 0) ntile = tile_rows_serial<G>(T, p, I, cur, end, [](int) { return 0; }, false);
    } else if (nw) {
        for (int w = lane; w < nw; w += 32) bm[w] = 0u;
        __syncwarp();
#pragma unroll
        for (int m = 0; m < G::TBM; ++m)
            for (int e = cur[m] + lane; e < end[m]; e += 32) {
                const int j = T.mcol[e] - lo;
                atomicOr(&bm[j >> 5], 1u << (j & 31));
            }
        __syncwarp();
        // exclusive prefix of the words' popcounts
        int carry = 0;
        for (int w0 = 0; w0 < nw; w0 += 32) {
            const int w = w0 + lane;
            const int c = w < nw ? __popc(bm[w]) : 0;
            int x = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (w < nw) wr[w] = carry + x - c;
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        __syncwarp();
        ntile = (carry + G::TBN - 1) / G::TBN;
    }
    if (lane == 0) cnt_s[wq] = ntile;
    __syncthreads();
    int total = 0;
#pragma unroll
    for (int k = 0; k < kTileRowWarps; ++k) total += cnt_s[k];
    if (wq == 0) {
        const int first = lookback_sum(T.look, bid, total, T.flags + 3, T.look_polls);
        if (lane == 0) {
            sh_base = first;
            if (bid == (int)gridDim.x - 1) T.flags[2] = first + total;
        }
    }
    __syncthreads();
    // tile q of this super-row: after the first q of each of the CTA's super-rows
    // and the q-th of those before it
    auto place = [&](int q) {
        int at = sh_base;
#pragma unroll
        for (int k = 0; k < kTileRowWarps; ++k) at += min(cnt_s[k], q) + (k < wq && cnt_s[k] > q ? 1 : 0);
        return at;
    };
    if (serial) {
        if (lane == 0) tile_rows_serial<G>(T, p, I, cur, end, place, true);
        return;
    }
    for (int q = lane; q < ntile; q += 32) {
        int *d = T.tiles + (size_t)place(q) * G::kTileInts;
        d[0] = p; d[1] = I; d[2] = -1; d[3] = 0;
        for (int k = 4; k < G::kTileInts; ++k) d[k] = -1;
    }
    __syncwarp();
    if (nw == 0) return;
#pragma unroll
    for (int m = 0; m < G::TBM; ++m)
        for (int e = cur[m] + lane; e < end[m]; e += 32) {
            const int jc = T.mcol[e];
            const int j = jc - lo;
            const int r = wr[j >> 5] + __popc(bm[j >> 5] & ((1u << (j & 31)) - 1u));
            int *d = T.tiles + (size_t)place(r / G::TBN) * G::kTileInts;
            d[4 + m * G::TBN + r % G::TBN] = e;
            d[G::kColOff + r % G::TBN] = jc;
        }
}

// the serial TBM-way merge (same tile order as the bitmap path)
template <class G, class Place>
__device__ int tile_rows_serial(const TileBuild &T, int p, int I, const int *cur0, const int *end0, const Place &place,
                                bool fill) {
    int cur[G::TBM], end[G::TBM];
    for (int m = 0; m < G::TBM; ++m) { cur[m] = cur0[m]; end[m] = end0[m]; }
    // the distinct columns needed by the TBM rows, in increasing order, are
    // packed TBN at a time into tiles: every tile column is needed by at least
    // one row
    int ncol = 0, n = 0;
    int *d = nullptr;
    // list heads kept in registers: one load per advance
    int head[G::TBM];
#pragma unroll
    for (int m = 0; m < G::TBM; ++m) head[m] = cur[m] < end[m] ? T.mcol[cur[m]] : 0x7fffffff;
    while (true) {
        int jmin = 0x7fffffff;
#pragma unroll
        for (int m = 0; m < G::TBM; ++m) jmin = min(jmin, head[m]);
        if (jmin == 0x7fffffff) break;
        const int c = ncol % G::TBN;
        if (c == 0) {
            if (fill) {
                d = T.tiles + (size_t)place(n) * G::kTileInts;
                d[0] = p; d[1] = I; d[2] = -1; d[3] = 0;
                for (int q = 4; q < G::kTileInts; ++q) d[q] = -1;
            }
            ++n;
        }
        if (fill) d[G::kColOff + c] = jmin;
#pragma unroll
        for (int m = 0; m < G::TBM; ++m)
            if (head[m] == jmin) {
                if (fill) d[4 + m * G::TBN + c] = cur[m];
                ++cur[m];
                head[m] = cur[m] < end[m] ? T.mcol[cur[m]] : 0x7fffffff;
            }
        ++ncol;
    }
    return n;
}

// one thread per tile: K-steps = union over the tile's A rows intersected with
// the union over its B rows, for each term (count, or fill at w)
template <class G>
__device__ int tile_steps_serial(const TileBuild &T, int t, int64_t w, bool fill) {
    const int *d = T.tiles + (size_t)t * G::kTileInts;
    const int p = d[0], I = d[1];
    const Job &job = T.jt.job[p];
    int n = 0;
    for (int term = 0; term < job.nterm; ++term) {
        const int am = job.a[term], bm = job.b[term];
        int cur[G::kSlots], end[G::kSlots];
        for (int q = 0; q < G::TBM; ++q) {
            const int i = G::TBM * I + q;
            cur[q] = end[q] = 0;
            if (i < T.NB) { cur[q] = T.rp[am * T.NB + i]; end[q] = T.rp[am * T.NB + i + 1]; }
        }
        for (int q = 0; q < G::TBN; ++q) {
            const int j = d[G::kColOff + q];
            cur[G::TBM + q] = end[G::TBM + q] = 0;
            if (j >= 0) { cur[G::TBM + q] = T.rp[bm * T.NB + j]; end[G::TBM + q] = T.rp[bm * T.NB + j + 1]; }
        }
        // list heads kept in registers: one load per advance
        int head[G::kSlots];
#pragma unroll
        for (int q = 0; q < G::kSlots; ++q) head[q] = cur[q] < end[q] ? T.col[cur[q]] : 0x7fffffff;
        while (true) {
            int kmin = 0x7fffffff;
#pragma unroll
            for (int q = 0; q < G::kSlots; ++q) kmin = min(kmin, head[q]);
            if (kmin == 0x7fffffff) break;
            bool anyA = false, anyB = false;
            int idx[G::kSlots];
#pragma unroll
            for (int q = 0; q < G::kSlots; ++q) {
                idx[q] = -1;
                if (head[q] == kmin) {
                    idx[q] = cur[q];
                    ++cur[q];
                    head[q] = cur[q] < end[q] ? T.col[cur[q]] : 0x7fffffff;
                    if (q < G::TBM) anyA = true; else anyB = true;
                }
            }
            if (anyA && anyB) {
                if (fill && w + n < T.cap_steps) {
                    int *s = T.steps + (size_t)(w + n) * G::kSlots;
                    for (int q = 0; q < G::kSlots; ++q) s[q] = idx[q] >= 0 && T.tpos ? T.tpos[idx[q]] : idx[q];
                }
                ++n;
            }
        }
        if (!fill && term == 0) T.tiles[(size_t)t * G::kTileInts + 2] = n;
    }
    return n;
}

// room for the n K-steps of tile t: their place, and the tile's record
template <class G>
__device__ __forceinline__ int64_t take_steps(const TileBuild &T, int t, int n) {
    const int64_t w = (int64_t)atomicAdd(reinterpret_cast<unsigned long long *>(T.flags + 4), (unsigned long long)n);
    const bool room = w + n <= T.cap_steps;
    if (!room) T.flags[1] = 1;
    T.step_rng[2 * (size_t)t] = w;
    T.step_rng[2 * (size_t)t + 1] = w + n;
    T.tiles[(size_t)t * G::kTileInts + 3] = room ? n : -1;
    return w;
}

// K-steps of one tile, one CTA per tile: per term, the columns k of the tile's
// TBM A rows and of its TBN B rows are marked in two shared-memory bitmaps
// over the window where both can have columns; a K-step is a k marked in
// both, its index the rank of k among those (prefix popcounts).  Each list
// entry at such a k writes its block index into its slot of the step; the
// other slots stay -1 (zero block).  Same steps, same order as the serial
// merge, which thread 0 runs for windows wider than the bitmaps.  A tile takes
// the room for its steps from a counter as it has counted them: where its
// list lies among the others' is left open, what is in it is not.  The kernel
// waits for loads, so a tile's slots are spread over four warps (one warp per
// tile took 25 us for the ~180 tiles of a 150-atom cluster), and counts and
// fills in one launch (count, scan and fill in three: 26 us there and 145 us for
// the 30,000 tiles of a 2,000-atom cluster, 12 and 112 us in one).
constexpr int kStepWarps = 4, kStepWords = 512;    // 16,384 columns per window
template <class G>
__global__ void __launch_bounds__(32 * kStepWarps) k_tile_steps(TileBuild T) {
    __shared__ unsigned ba[2][kStepWords], bb[kStepWords];
    __shared__ int wr[2][kStepWords];
    __shared__ int cur[2][G::kSlots], end[2][G::kSlots], lo_c[2][G::kSlots], hi_c[2][G::kSlots];
    __shared__ int sh_n[2];
    __shared__ int64_t sh_w;
    static_assert(2 * G::kSlots <= 32 * kStepWarps, "one thread per slot and term");
    const int tid = threadIdx.x, wq = tid >> 5, lane = tid & 31;
    if (T.flags[3]) {
        if (blockIdx.x == 0 && tid == 0) T.flags[1] = 1;
        return;
    }
    const int ntile = T.flags[2];
    for (int t = blockIdx.x; t < ntile; t += gridDim.x) {
        const int *d = T.tiles + (size_t)t * G::kTileInts;
        const int p = d[0], I = d[1];
        const Job &job = T.jt.job[p];
        if (tid < job.nterm * G::kSlots) {
            const int term = tid / G::kSlots, q = tid % G::kSlots;
            const int mat = q < G::TBM ? job.a[term] : job.b[term];
            const int row = q < G::TBM ? G::TBM * I + q : d[G::kColOff + q - G::TBM];
            int c = 0, e = 0, l = 0x7fffffff, h = -1;
            if (row >= 0 && row < T.NB) {
                c = T.rp[mat * T.NB + row];
                e = T.rp[mat * T.NB + row + 1];
                if (c < e) {
                    l = T.col[c];
                    h = T.col[e - 1];
                }
            }
            cur[term][q] = c;
            end[term][q] = e;
            lo_c[term][q] = l;
            hi_c[term][q] = h;
        }
        __syncthreads();
        // the window of every term must fit the bitmaps, else the serial merge
        int lo_t[2], hi_t[2];
        bool fits = true;
#pragma unroll
        for (int term = 0; term < 2; ++term) {
            lo_t[term] = 0;
            hi_t[term] = -1;
            if (term >= job.nterm) continue;
            int loA = 0x7fffffff, hiA = -1, loB = 0x7fffffff, hiB = -1;
            for (int q = 0; q < G::TBM; ++q) {
                loA = min(loA, lo_c[term][q]);
                hiA = max(hiA, hi_c[term][q]);
            }
            for (int q = G::TBM; q < G::kSlots; ++q) {
                loB = min(loB, lo_c[term][q]);
                hiB = max(hiB, hi_c[term][q]);
            }
            lo_t[term] = max(loA, loB);
            hi_t[term] = min(hiA, hiB);
            if (hi_t[term] >= lo_t[term] && ((hi_t[term] - lo_t[term]) >> 5) + 1 > T.max_words) fits = false;
        }
        if (!fits) {
            if (tid == 0) {
                const int n = tile_steps_serial<G>(T, t, 0, false);
                tile_steps_serial<G>(T, t, take_steps<G>(T, t, n), true);
            }
            __syncthreads();
            continue;
        }
        // the steps of each term
#pragma unroll
        for (int term = 0; term < 2; ++term) {
            const int lo = lo_t[term], hi = hi_t[term];
            const int nw = hi >= lo ? ((hi - lo) >> 5) + 1 : 0;
            unsigned *both_w = ba[term];
            for (int x = tid; x < nw; x += 32 * kStepWarps) { both_w[x] = 0u; bb[x] = 0u; }
            __syncthreads();
            if (nw)
                for (int q = wq; q < G::kSlots; q += kStepWarps) {
                    unsigned *bmap = q < G::TBM ? both_w : bb;
                    const int qe = end[term][q];
                    for (int e = cur[term][q] + lane; e < qe; e += 32) {
                        const int k = T.col[e];
                        if (k < lo || k > hi) continue;
                        atomicOr(&bmap[(k - lo) >> 5], 1u << ((k - lo) & 31));
                    }
                }
            __syncthreads();
            if (wq == 0) {
                int carry = 0;
                for (int x0 = 0; x0 < nw; x0 += 32) {
                    const int x = x0 + lane;
                    unsigned both = 0u;
                    if (x < nw) {
                        both = both_w[x] & bb[x];
                        both_w[x] = both;
                    }
                    const int c = __popc(both);
                    int y = c;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int z = __shfl_up_sync(0xffffffffu, y, o);
                        if (lane >= o) y += z;
                    }
                    if (x < nw) wr[term][x] = carry + y - c;
                    carry += __shfl_sync(0xffffffffu, y, 31);
                }
                if (lane == 0) {
                    sh_n[term] = carry;
                    if (term == 0) T.tiles[(size_t)t * G::kTileInts + 2] = carry;
                    else sh_w = take_steps<G>(T, t, sh_n[0] + carry);
                }
            }
            __syncthreads();
        }
        // -1 everywhere, then the stored blocks (nothing without room for all)
        const int n0 = sh_n[0], n = n0 + sh_n[1];
        const int64_t w = sh_w;
        if (w + n <= T.cap_steps) {
            for (int q = tid; q < n * G::kSlots; q += 32 * kStepWarps) T.steps[(size_t)w * G::kSlots + q] = -1;
            __syncthreads();
#pragma unroll
            for (int term = 0; term < 2; ++term) {
                const int lo = lo_t[term], hi = hi_t[term];
                if (hi < lo) continue;
                const int64_t at = w + (term ? n0 : 0);
                for (int q = wq; q < G::kSlots; q += kStepWarps) {
                    const int qe = end[term][q];
                    for (int e = cur[term][q] + lane; e < qe; e += 32) {
                        const int k = T.col[e];
                        if (k < lo || k > hi) continue;
                        const int kk = k - lo;
                        const unsigned word = ba[term][kk >> 5];
                        if (!((word >> (kk & 31)) & 1u)) continue;
                        const int r = wr[term][kk >> 5] + __popc(word & ((1u << (kk & 31)) - 1u));
                        T.steps[(size_t)(at + r) * G::kSlots + q] = T.tpos ? T.tpos[e] : e;
                    }
                }
            }
        }
        __syncthreads();
    }
}

template <class G>
TcPlan build_plan(const MatSet &in, const JobTable &jt, const SysDev &sd, const int *out_rp, const int *mcol,
                  TcWork &w, JobMask job_mask, int unit0, int unit1, int64_t nupper, int64_t min_steps,
                  cudaStream_t st) {
    TcPlan plan{};
    const int NB = in.NB, NBT = (NB + G::TBM - 1) / G::TBM;
    const int nrowt = unit1 - unit0;
    const int rgrid = std::max(0, (nrowt + kTileRowWarps - 1) / kTileRowWarps);
    if (nrowt <= 0 || nupper <= 0) return plan;
    // every tile of a super-row but its last one has TBN columns, each with at
    // least one upper slot
    const int64_t max_tile = nupper / G::TBN + nrowt;
    plan.max_tile = (int)max_tile;
    w.tiles.ensure((size_t)max_tile * G::kTileInts);
    w.step_rng.ensure(2 * (size_t)max_tile);
    w.steps.ensure((size_t)std::max<int64_t>(min_steps, 1) * G::kSlots);
    plan.cap_steps = (int64_t)(w.steps.cap / G::kSlots);
    // test settings, each for one plan
    const int inject = w.knobs.inject & (kInjectTileWait | kInjectStepRoom);
    w.knobs.inject &= ~inject;
    if (inject & kInjectStepRoom) plan.cap_steps = 1;
    TileBuild T{};
    T.rp = in.row_ptr.p; T.col = in.col.p; T.NB = NB; T.NBT = NBT; T.jt = jt;
    T.out_rp = out_rp; T.mcol = mcol; T.sys_of_row = sd.sys_of_row.p; T.active = sd.active.p;
    T.job_mask = job_mask;
    T.u0 = unit0; T.u1 = unit1;
    T.sys_tier = sd.tier.p;
    T.look = reinterpret_cast<unsigned long long *>(w.counters + 8);
    T.look_polls = inject & kInjectTileWait ? 0 : kLookPolls;
    T.tpos = w.tpos_valid ? w.tpos.p : nullptr;
    T.tiles = w.tiles.p; T.step_rng = w.step_rng.p; T.steps = w.steps.p;
    T.cap_steps = plan.cap_steps; T.flags = w.counters;
    static_assert(kTileRowWords == kStepWords, "one window bound for both plan builders");
    T.max_words = w.knobs.window_words > 0 && w.knobs.window_words < kTileRowWords ? w.knobs.window_words
                                                                                    : kTileRowWords;
    const int sgrid = (int)std::min<int64_t>(max_tile, 152 * 16);
    k_tile_rows<G><<<rgrid, 32 * kTileRowWarps, 0, st>>>(T);
    RDM_LAUNCH_CHECK();
    k_tile_steps<G><<<sgrid, 32 * kStepWarps, 0, st>>>(T);
    RDM_LAUNCH_CHECK();
    return plan;
}

}  // namespace
}  // namespace rdm

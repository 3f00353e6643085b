"""Tile lists, K-step lists and the compaction's pattern of long, thin block
matrices: their offsets are prefix sums across the CTAs of one launch (8 rows
or super-rows each, 32 CTAs looked at in one go), and the K-step lists start in
room guessed from the number of block pairs.  Entries are small integers, so
every arithmetic gives the exact product."""

import numpy as np
import pytest
import scipy.sparse as sp

from synth import Bsr, System

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rdm():
    from paper_2009_03551_gb300 import build as b
    b.build()
    from paper_2009_03551_gb300 import rdm as mod
    return mod


def band(rng, nb, b, off):
    """Symmetric matrix with the block diagonals 0 and +-off, integer entries."""
    i = np.arange(nb)
    d = rng.integers(-2, 3, (nb, b, b)).astype(float)
    u = rng.integers(-2, 3, (max(nb - off, 0), b, b)).astype(float) if off else np.zeros((0, b, b))
    k = i[:len(u)]
    rows = np.concatenate([i, k, k + off])
    cols = np.concatenate([i, k + off, k])
    vals = np.concatenate([d + d.transpose(0, 2, 1), u, u.transpose(0, 2, 1)])
    o = np.lexsort((cols, rows))
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=nb))]).astype(np.int32)
    return rp, cols[o].astype(np.int32), np.ascontiguousarray(vals[o])


@pytest.mark.parametrize("nb,b,off,mode", [
    (1, 2, 0, "fp64"), (8, 2, 1, "fp64"), (9, 4, 2, "fp64"),              # one CTA, two
    (256, 2, 1, "fp64"), (257, 4, 3, "fp64"), (8400, 2, 7, "fp64"),       # 32, 33 and 1,050 CTAs of the compaction
    (2047, 16, 3, "mixed_fp16"), (2112, 16, 1, "mixed_bf16"),             # 32 and 33 CTAs of the tile list
    (521, 64, 2, "mixed_bf16"), (1100, 32, 1, "mixed_fp16"), (1100, 32, 5, "fp64"),
    (95000, 16, 0, "mixed_fp16"),      # one pair per K-step: more steps than the first guess has room for
])
def test_lists_of_long_matrices(rdm, nb, b, off, mode):
    rng = np.random.default_rng(nb + b)
    rp, ci, va = band(rng, nb, b, off)
    n = nb * b
    A = Bsr(nb, b, n, rp, ci, va)
    S = sp.bsr_matrix((va, ci, rp), shape=(n, n))
    exact = sp.bsr_matrix(S @ S + 2.0 * S, blocksize=(b, b))
    exact.sort_indices()
    # a threshold inside the widest gap between the middle half of the block norms
    nrm = np.sqrt((exact.data ** 2).sum((1, 2)))
    mid = np.sort(nrm)[len(nrm) // 4:max(3 * len(nrm) // 4, 2)]
    k = int(np.argmax(np.diff(mid))) if off else 0
    tau = float(0.5 * (mid[k] + mid[k + 1])) if off else 0.0
    keep = nrm >= tau
    row = np.repeat(np.arange(nb), np.diff(exact.indptr))
    h = rdm.rdm_create(0)
    try:
        got = rdm.rdm_block_product(h, A, None, A, 2.0, 1.0, 1, tau, rdm.MODES[mode])
    finally:
        rdm.rdm_destroy(h)
    assert np.array_equal(got.row_ptr, np.concatenate([[0], np.cumsum(np.bincount(row[keep], minlength=nb))]))
    assert np.array_equal(got.col_idx, exact.indices[keep])
    assert np.array_equal(got.vals, exact.data[keep])


def test_a_step_whose_lists_outgrow_their_room_is_repeated(rdm):
    """A block-diagonal H0 of 95,000 blocks has one pair to a K-step: the first
    step's list does not fit, which the host learns after the copy into the next
    step's matrices was launched.  Every block of P0 is the projector of its
    block of H0 (split fp16 ladder at tol 1e-8: 1e-5 is far above its error and
    far below a missing or misplaced step)."""
    nb, b, nocc = 95000, 16, 5
    rng = np.random.default_rng(3)
    q, _ = np.linalg.qr(rng.standard_normal((b, b)))
    ev = np.concatenate([np.linspace(-2.0, -1.0, nocc), np.linspace(1.0, 2.0, b - nocc)])
    blk = (q * ev) @ q.T
    blk = 0.5 * (blk + blk.T)
    i = np.arange(nb, dtype=np.int32)
    h0 = Bsr(nb, b, nb * b, np.arange(nb + 1, dtype=np.int32), i, np.tile(blk, (nb, 1, 1)))
    s = System("blocks", "diagonal", np.zeros((nb, 3)), b, nocc * nb, b, h0, [], (), 0.0, 3)
    sol = rdm.Solver(0)
    sol.set_params(tau=1e-7, tol=1e-8, mode="mixed_fp16", max_iter=60)
    sol.load(s)
    code, info = sol.solve()
    assert code == rdm.RDM_OK
    p0 = sol.p0()
    assert np.array_equal(p0.col_idx, i)
    assert np.max(np.abs(p0.vals - q[:, :nocc] @ q[:, :nocc].T)) <= 1e-5


@pytest.mark.parametrize("mode", ["fp64", "mixed_fp16"])
def test_solve_with_little_memory(rdm, mode):
    """With three quarters of the memory that a solve takes when it has all it
    wants, it goes on without its optional buffers: the split ladder to the same
    bits (the copies it does without hold the same numbers), the FP64 mode to the
    rounding of its products (1e-16 each, amplified by at most 2^20)."""
    import torch
    from synth import make_cluster
    s = make_cluster(600, opa=8, b=32, cutoff=10.0, seed=4, dirs=("x",))

    def solve():
        sol = rdm.Solver(0)
        sol.set_params(tau=1e-6, tol=1e-9, mode=mode, max_iter=60)
        sol.load(s)
        code, info = sol.solve()
        assert code == rdm.RDM_OK
        p1 = sol.p1(0, 0)
        peak = info.device_bytes_peak
        sol.close()
        return p1, peak

    ref, peak = solve()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    hold = [torch.empty(int(free - 0.75 * peak) >> 20, 1 << 20, dtype=torch.uint8, device="cuda")]
    try:
        got, less = solve()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert less < peak
    if mode == "fp64":
        assert np.array_equal(got.row_ptr, ref.row_ptr)
        assert np.max(np.abs(got.vals - ref.vals)) <= 1e-9 * np.max(np.abs(ref.vals))
    else:
        assert np.array_equal(got.col_idx, ref.col_idx) and np.array_equal(got.vals, ref.vals)

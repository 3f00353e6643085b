"""The mask of a product whose inputs are symmetric only to the uploads'
tolerance (1e-12 of the largest element): a block whose bound reaches the
threshold while its mirror's does not is in the mask with its mirror, so that
the compaction finds both.  The inputs have one occupied orbital per block row,
so that bounds and norms of the blocks in question are equal."""

import numpy as np
import pytest

from synth import Bsr, System

TAU = 1e-6
# (row, column, the smaller element is the lower one): X1 elements of
# HI tau / 2 and LO tau / 2 at mirrored places.  The first step adds the two (a
# product takes B_kj from block (j, k)): a norm of (1 + 7e-4) tau, while the bounds
# are HI tau and LO tau and the symbolic phase keeps those above (1 - 2^-10) tau
HI, LO = 1 + 3e-3, 1 - 1.6e-3
PAIRS = [(1, 4, True), (2, 3, False), (0, 5, True), (6, 7, False)]
NB = 8
BIG = 1e4


def inputs(b):
    """Block-diagonal H0 = diag(-1, 1, .., 1) per block (X0 = diag(1, 0, .., 0)
    from the start) and H1 with the elements of PAIRS at orbital 0 of their
    blocks, and a large virtual-virtual element that sets the tolerance."""
    d = np.ones(b)
    d[0] = -1.0
    i = np.arange(NB, dtype=np.int32)
    h0 = Bsr(NB, b, NB * b, np.arange(NB + 1, dtype=np.int32), i, np.tile(np.diag(d), (NB, 1, 1)))
    el = {(0, 0): (BIG, 1)}
    for r, c, lower in PAIRS:
        hi, lo = -TAU * HI, -TAU * LO         # X1 = -H1 / 2
        el[(r, c)], el[(c, r)] = ((hi if lower else lo), 0), ((lo if lower else hi), 0)
    keys = sorted(el)
    va = np.zeros((len(keys), b, b))
    for q, k in enumerate(keys):
        va[q, el[k][1], el[k][1]] = el[k][0]
    rp = np.searchsorted([k[0] for k in keys], np.arange(NB + 1)).astype(np.int32)
    h1 = Bsr(NB, b, NB * b, rp, np.array([k[1] for k in keys], dtype=np.int32), va)
    return System("asym", "test", np.zeros((NB, 3)), b, NB, b, h0, [h1], ("x",), 0.0, 0), el


def test_the_inputs_have_unequal_bounds():
    """Without the larger norm of both blocks the bounds of a pair lie on either
    side of the threshold, and the difference passes the check of the uploads."""
    _, el = inputs(16)
    for r, c, _ in PAIRS:
        n = {}
        for k in ((r, c), (c, r)):
            x = np.float64(abs(el[k][0]) / 2)
            f = np.float32(x)
            n[k] = float(f if f >= x else np.nextafter(f, np.float32(1)))
        bound = sorted(2.0 * v for v in n.values())
        assert bound[0] < TAU * (1 - 2.0 ** -10) and bound[1] >= TAU
        assert abs(el[(r, c)][0] - el[(c, r)][0]) <= 1e-12 * BIG


@pytest.fixture(scope="module")
def rdm():
    from paper_2009_03551_gb300 import build as b
    b.build()
    from paper_2009_03551_gb300 import rdm as mod
    return mod


@pytest.mark.gpu
@pytest.mark.parametrize("b,mode", [(16, "mixed_bf16"), (32, "mixed_bf16"), (64, "mixed_bf16"), (8, "fp64"),
                                    (32, "fp64"), (32, "fp32")])
def test_blocks_of_unequal_bounds_come_with_their_mirrors(rdm, b, mode):
    """One step, X1 <- X0 X1 + X1 X0: every pair is kept, as a block and its
    transpose (tolerance: the 16-bit operands of the bf16 split, 2^-15)."""
    s, el = inputs(b)
    sol = rdm.Solver(0)
    sol.set_params(tau=TAU, tol=0.0, mode=mode, max_iter=1)
    sol.load(s)
    rdm.rdm_force_branches(sol.h, [1])
    code, info = sol.solve()
    assert code == rdm.RDM_NOT_CONVERGED and info.iterations == 1
    got = sol.p1(0, 0).to_dense()
    want = np.zeros_like(got)
    for r, c, _ in PAIRS:
        want[r * b, c * b] = want[c * b, r * b] = -0.5 * (el[(r, c)][0] + el[(c, r)][0])
    assert np.array_equal(got != 0, want != 0)
    assert np.max(np.abs(got - want)) <= 2.0 ** -15 * TAU
    sol.close()


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["fp64", "mixed_bf16"])
def test_block_product_with_an_unequal_linear_term(rdm, mode):
    """C = X + 0 A A: the mask follows the bounds of X alone, and a pair is kept
    where its upper block reaches tau."""
    s, el = inputs(32)
    h = rdm.rdm_create(0)
    try:
        got = rdm.rdm_block_product(h, s.h0, None, s.h1[0], 1.0, 0.0, 1, TAU, rdm.MODES[mode]).to_dense()
    finally:
        rdm.rdm_destroy(h)
    want = np.zeros_like(got)
    want[1, 1] = BIG
    for r, c, lower in PAIRS:
        if lower:
            want[r * 32, c * 32] = want[c * 32, r * 32] = el[(r, c)][0]
    assert np.array_equal(got != 0, want != 0)
    assert np.allclose(got, want, rtol=2.0 ** -22, atol=0.0)           # the linear term is FP32 in the split

"""FP64 solves of 32 x 32 blocks with a truncation threshold run their products
on the tensor cores as exact sums of 8-slice products (128 x 64 tiles: 4 block
rows x 2 block columns).  Checked against the stepwise oracle at the edges of
the tiles, and against the FP64 FMA chains of the same solve at 16 x 16 blocks,
which stay on the CUDA cores."""

import numpy as np
import pytest

from blockcheck import max_rel_err
from oracle import tc2_response
from oracle.dense import rel_frobenius
from synth import make_cluster

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rdm():
    from paper_2009_03551_gb300 import build as b
    b.build()
    from paper_2009_03551_gb300 import rdm as mod
    return mod


# 1, 2, 4, 5 and 9 block rows (one tile row is 4, one tile column 2), the last
# block full or ragged; no, one and three field directions
@pytest.mark.parametrize("atoms,dirs", [(4, "xyz"), (7, ""), (13, "x"), (17, "xyz"), (33, "xyz")])
def test_fp64_slice_products_follow_the_stepwise_oracle(rdm, atoms, dirs):
    s = make_cluster(atoms, opa=8, b=32, cutoff=10.0, seed=atoms, dirs=tuple(dirs))
    h1s = [m.to_dense() for m in s.h1]
    ob = tc2_response(s.h0.to_dense(), h1s, s.n_occ, s.b, tau=1e-6, tol=1e-9)
    sol = rdm.Solver(0)
    sol.set_params(tau=1e-6, tol=0.0, mode="fp64", max_iter=ob.iterations)
    sol.load(s)
    rdm.rdm_force_branches(sol.h, ob.branches)
    code, info = sol.solve()
    assert code in (rdm.RDM_OK, rdm.RDM_NOT_CONVERGED) and info.iterations == ob.iterations
    assert info.kernel_flops[1] > 0
    # same filter, same steps: what differs is rounding (1e-16 per product,
    # grown by at most 2 per step of the ~20 doublings of the spectrum's edges)
    assert rel_frobenius(sol.p0().to_dense(), ob.p0) <= 1e-10
    assert max_rel_err(sol.p0().to_dense(), ob.p0) <= 1e-10
    for d in range(len(dirs)):
        got = sol.p1(0, "xyz".index(dirs[d])).to_dense()
        assert rel_frobenius(got, ob.p1s[d]) <= 1e-10
        assert max_rel_err(got, ob.p1s[d]) <= 1e-10
        assert np.array_equal(got, got.T)


def test_slices_need_a_threshold(rdm):
    """At tau = 0 every block is wanted, however small: the products stay FP64
    FMA chains, as at b = 16; just above the bound the slices run.  P0 agrees
    far below the threshold either way."""
    s = make_cluster(17, opa=8, b=32, cutoff=10.0, seed=2, dirs=("x",))
    out = {}
    for tau in (0.0, 1e-11, 2e-10):
        sol = rdm.Solver(0)
        sol.set_params(tau=tau, tol=1e-9, mode="fp64", max_iter=60)
        sol.load(s)
        code, info = sol.solve()
        assert code == rdm.RDM_OK
        out[tau] = (sol.p0().to_dense(), info.simt_launches)
    assert out[0.0][1] > 0 and out[1e-11][1] > 0 and out[2e-10][1] == 0
    for tau in (1e-11, 2e-10):
        assert rel_frobenius(out[tau][0], out[0.0][0]) <= 1e-9


@pytest.mark.parametrize("tau,tau_x1", [(1e-6, 0.0), (0.0, 1e-6)])
def test_accounting_of_thresholds_on_either_side_of_the_bound(rdm, tau, tau_x1):
    """X0^2 as slices and X1's products as FP64 FMAs, and the other way round:
    both count as FP64 products, in flops and in time, and the FMA chains
    appear among the issued ones."""
    s = make_cluster(17, opa=8, b=32, cutoff=10.0, seed=2, dirs=("x", "y"))
    info = {}
    for dirs in (0, 2):
        y = type(s)(**{**s.__dict__, "h1": s.h1[:dirs], "dirs": s.dirs[:dirs]})
        sol = rdm.Solver(0)
        sol.set_params(tau=tau, tau_x1=tau_x1, tol=0.0, mode="fp64", max_iter=12)
        sol.load(y)
        code, info[dirs] = sol.solve()
        assert code == rdm.RDM_NOT_CONVERGED and info[dirs].iterations == 12
        sol.close()
    i0, i2 = info[0], info[2]
    assert i2.oz_launches > 0 and i2.simt_launches > 0
    assert i2.kernel_flops[1] == i2.useful_flops and i2.kernel_flops[4] == 0
    assert i2.kernel_ms[2] > 0 and i2.kernel_ms[7] == 0
    # X0's recursion does not depend on X1: the FMA part is issued as it is useful
    if tau > 0:
        assert i2.issued_flops - i0.issued_flops == i2.useful_flops - i0.useful_flops
    else:
        assert i0.issued_flops == i0.useful_flops < i2.issued_flops - (i2.useful_flops - i0.useful_flops)

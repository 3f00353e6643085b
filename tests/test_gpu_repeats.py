"""Steps that have to be done again: a wait between the CTAs of a prefix sum runs
out (tile lists, compaction), or the K-step lists outgrow their room.  Each
happens on request, once, in a step whose result is not waited for (the copy
into the next step's matrices and their statistics are then launched before the
host knows) and, with the products in groups, in one that is.  The repeated step
gives the same bits."""

import numpy as np
import pytest

from synth import make_cluster

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rdm():
    from paper_2009_03551_gb300 import build as b
    b.build()
    from paper_2009_03551_gb300 import rdm as mod
    return mod


def solve(rdm, s, inject=0, **prm):
    sol = rdm.Solver(0)
    sol.set_params(tau=1e-6, tol=1e-9, max_iter=60, **prm)
    sol.load(s)
    rdm.rdm_set_test_knobs(sol.h, inject=inject)
    code, info = sol.solve()
    assert code == rdm.RDM_OK
    out = [sol.p0()] + [sol.p1(0, d) for d in range(3)]
    sol.close()
    return out, info


@pytest.fixture(scope="module")
def system():
    return make_cluster(75, opa=8, b=16, cutoff=10.0, seed=5)


# the injected failures: tile lists 1, compaction 2, K-steps 4, and all at once;
# 38 uploaded rows of 16 (blocks of 32: 19 rows, 20 super-rows of 4 with 4 jobs,
# about 10 of them in the 384 blocks of a group of 3 MiB; a wait takes more than 8)
@pytest.mark.parametrize("inject", [1, 2, 4, 7])
@pytest.mark.parametrize("prm", [
    dict(mode="mixed_fp16", block_size=32), dict(mode="mixed_bf16", block_size=16), dict(mode="fp64", block_size=32),
    dict(mode="mixed_fp16", block_size=32, chunk_mb=3), dict(mode="fp64", block_size=32, chunk_mb=3),
], ids=["split32", "split16", "slices", "split32-groups", "slices-groups"])
def test_a_repeated_step_gives_the_same_bits(rdm, system, prm, inject):
    ref, i0 = solve(rdm, system, **prm)
    got, i1 = solve(rdm, system, inject=inject, **prm)
    assert (i0.product_groups > 1) == ("chunk_mb" in prm)
    assert i1.kernel_launches > i0.kernel_launches and i1.iterations == i0.iterations
    for r, g in zip(ref, got):
        assert np.array_equal(r.row_ptr, g.row_ptr) and np.array_equal(r.col_idx, g.col_idx)
        assert np.array_equal(r.vals, g.vals)

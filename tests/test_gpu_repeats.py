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


@pytest.mark.parametrize("mode,b", [("mixed_fp16", 32), ("mixed_bf16", 16), ("fp32", 32)])
def test_a_step_without_memory_is_repeated_without_its_optional_buffers(rdm, system, mode, b):
    """Whichever allocation of a step fails, the results keep their bits."""
    ref, i0 = solve(rdm, system, mode=mode, block_size=b)
    for k in range(1, 60, 2):
        got, i1 = solve(rdm, system, inject=8 * k, mode=mode, block_size=b)
        assert i1.iterations == i0.iterations
        for r, g in zip(ref, got):
            assert np.array_equal(r.col_idx, g.col_idx) and np.array_equal(r.vals, g.vals), k


def test_an_fp64_solve_has_one_arithmetic(rdm, system):
    """FP64 mode at 32 x 32 blocks: slices, or FMA chains where the caller asks
    for them or where a step with slices finds no memory, in every step of the
    solve; the info tells which."""
    slices, i0 = solve(rdm, system, mode="fp64", block_size=32)
    fma, i1 = solve(rdm, system, mode="fp64", block_size=32, refine_x0=1)
    assert i0.oz_launches > 0 and i0.simt_launches == 0
    assert i1.oz_launches == 0 and i1.simt_launches > 0
    failed = 0
    for k in range(1, 60, 2):
        got, i = solve(rdm, system, inject=8 * k, mode="fp64", block_size=32)
        assert (i.oz_launches > 0) != (i.simt_launches > 0)
        failed += i.oz_launches == 0
        for r, g in zip(slices if i.oz_launches else fma, got):
            assert np.array_equal(r.col_idx, g.col_idx) and np.array_equal(r.vals, g.vals), k
    assert failed > 10
    # rounding of either (1e-16 a product, doubled by each of ~20 steps)
    for r, g in zip(slices, fma):
        assert np.max(np.abs(r.to_dense() - g.to_dense())) <= 1e-9 * np.max(np.abs(g.vals))


@pytest.mark.parametrize("prm", [dict(correct=1), dict(split_directions=1)], ids=["correct", "directions"])
def test_solves_of_several_passes_start_again_as_a_whole(rdm, system, prm):
    """A pass after the first one that finds no room for its slices."""
    prm = dict(prm, mode="fp64", block_size=32)
    ref = {True: solve(rdm, system, **prm)[0], False: solve(rdm, system, refine_x0=1, **prm)[0]}
    seen = set()
    for k in range(3, 260, 16):
        got, i = solve(rdm, system, inject=8 * k, **prm)
        seen.add(i.oz_launches > 0)
        for r, g in zip(ref[i.oz_launches > 0], got):
            assert np.array_equal(r.col_idx, g.col_idx) and np.array_equal(r.vals, g.vals), k
    assert seen == {True, False}


def test_slice_plans_make_room_for_their_own_jobs(rdm):
    """The final tier's slice plan holds X0^2 alone, a small part of a step's
    pairs with three field directions: its lists, made for every pair at 24 bytes
    per two, held 38 of the 2,146 MB of this solve beyond what they need."""
    s = make_cluster(600, opa=8, b=32, cutoff=10.0, seed=4)
    _, info = solve(rdm, s, mode="mixed_fp16")
    assert 1.5e9 < info.device_bytes_peak <= 2.125e9


def test_uploads_give_back_what_the_next_problem_does_not_use(rdm):
    """A handle that held H1 matrices solves a system without them in the memory that
    a new handle takes."""
    s = make_cluster(400, opa=8, b=32, cutoff=10.0, seed=4)
    bare = type(s)(**{**s.__dict__, "h1": [], "dirs": ()})

    def peak(first):        # (of every handle of the process)
        sol = rdm.Solver(0)
        sol.set_params(tau=1e-6, tol=1e-9, mode="fp64", max_iter=60)
        if first is not None:
            sol.load(first)
        sol.load(bare)
        code, info = sol.solve()
        assert code == rdm.RDM_OK
        sol.close()
        return info.device_bytes_peak

    assert peak(s) == peak(None)


def test_products_between_solves(rdm, system):
    """A block product borrows the handle's page-locked memory: solves before and
    after it, and the product itself, are what they are on handles of their own."""
    ref, _ = solve(rdm, system, mode="mixed_fp16")
    h = rdm.rdm_create(0)
    want = rdm.rdm_block_product(h, system.h0, None, None, 0.0, 1.0, 1, 1e-6)
    rdm.rdm_destroy(h)
    sol = rdm.Solver(0)
    sol.set_params(tau=1e-6, tol=1e-9, max_iter=60, mode="mixed_fp16")
    sol.load(system)
    for _ in range(2):
        prod = rdm.rdm_block_product(sol.h, system.h0, None, None, 0.0, 1.0, 1, 1e-6)
        with pytest.raises(rdm.RdmError):       # a product that fails gives it back too
            rdm.rdm_block_product(sol.h, system.h0, system.h1[0], system.h0, 0.0, 1.0, 2, -1.0)
        code, _ = sol.solve()
        assert code == rdm.RDM_OK
        assert np.array_equal(prod.vals, want.vals)
        for r, g in zip(ref, [sol.p0()] + [sol.p1(0, d) for d in range(3)]):
            assert np.array_equal(r.vals, g.vals)
    sol.close()

"""Performance cases: the work that a program has this library do.

A program holds a system's Hamiltonian H0 and its field perturbations H1 as
block-sparse matrices on the GPU, hands them to a solver that it keeps
(``Solver.load``), solves, and reads the density matrix P0, the response
density matrices P1 and the polarizability back into pinned host buffers that
it keeps as well.  One pass of a case is that whole call.  The smallest case
is the allocation-free inner product of two block-sparse matrices, a call of
a few microseconds.

The systems are the synthetic gapped ones of this repository's workloads:
chains of equally spaced atoms, clusters and slabs packed at random at the
atom density of liquid water and ordered along a Morton curve, with hopping
blocks that decay exponentially and dipole perturbations.  They are drawn on
the GPU from the seed alone.
"""

import math

import torch

DENSITY = 0.0148        # atoms / bohr^3, liquid water
MIN_DIST = 2.5          # bohr, closest pair of a cluster or slab
SPACING = 2.8           # bohr, neighbours of a chain
THICKNESS = 30.0        # bohr, slab


def listed():
    return [
        # the reduction behind the polarizability as a call of its own, for a
        # program that may not allocate: the smallest call, launches and host
        dict(name="dot-150", do="dot", kind="cluster", atoms=150, opa=8, b=32),
        # the small exact workload: 64 atoms in 4 x 4 blocks, no truncation,
        # FP64, one field direction; many tiny products
        dict(name="chain-64-fp64-exact", do="solve", kind="chain", atoms=64, opa=4, b=4, mode="fp64", tau=0.0, dirs=1),
        # a small molecule in the default mixed-precision ladder: latency
        dict(name="cluster-150-fp16", do="solve", kind="cluster", atoms=150, opa=8, b=32, mode="mixed_fp16", tau=1e-6,
             dirs=3),
        # a long chain molecule: narrow band, few blocks per row, many rows
        dict(name="chain-1501-fp16", do="solve", kind="chain", atoms=1501, opa=8, b=32, mode="mixed_fp16", tau=1e-6,
             dirs=3),
        # atom blocks of 8 as a code stores them, products in 32 x 32 blocks,
        # one field direction
        dict(name="cluster-601-fp16-b8", do="solve", kind="cluster", atoms=601, opa=8, b=8, block_size=32,
             mode="mixed_fp16", tau=1e-6, dirs=1),
        # the FP64 mode, the accuracy reference of every study
        dict(name="cluster-300-fp64", do="solve", kind="cluster", atoms=300, opa=8, b=32, mode="fp64", tau=1e-6,
             dirs=3),
        # the FP32 mode
        dict(name="cluster-1000-fp32", do="solve", kind="cluster", atoms=1000, opa=8, b=32, mode="fp32", tau=1e-6,
             dirs=3),
        # a non-orthogonal basis: overlap matrix, its inverse square root by
        # Newton-Schulz products, transforms there and back
        dict(name="cluster-151-fp16-overlap", do="solve", kind="cluster", atoms=151, opa=8, b=32, mode="mixed_fp16",
             tau=1e-6, dirs=3, overlap=True),
        # the bf16 ladder with the accuracy correction of P0 and P1
        dict(name="cluster-250-bf16-correct", do="solve", kind="cluster", atoms=250, opa=8, b=32, mode="mixed_bf16",
             tau=1e-6, dirs=3, correct=True),
        # the bf16 ladder with a loose threshold, tightened in the final tier
        dict(name="cluster-2000-bf16", do="solve", kind="cluster", atoms=2000, opa=8, b=32, mode="mixed_bf16",
             tau=1e-5, tau_refine=1e-7, dirs=3),
        # independent systems of uneven size in one batch
        dict(name="batch-5-fp16", do="solve", kind="batch", atoms=300, atoms_to=1500, systems=5, opa=8, b=32,
             mode="mixed_fp16", tau=1e-6, dirs=3),
        # a solid: the largest
        dict(name="slab-5000-fp16", do="solve", kind="slab", atoms=5000, opa=8, b=32, mode="mixed_fp16", tau=1e-6,
             dirs=3),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    ladder = dict(opa=8, b=32, mode=rng.choice(["mixed_fp16", "mixed_fp16", "mixed_bf16"]),
                  tau=rng.choice([1e-5, 1e-6, 1e-6]), dirs=rng.choice([1, 3, 3]))
    what = rng.choice(["dot", "exact", "fp64", "fp32", "cluster", "cluster", "slab", "chain", "batch", "atom blocks",
                       "blocks", "overlap", "correct"])
    if what == "dot":
        return dict(do="dot", kind=rng.choice(["chain", "cluster", "slab"]), atoms=size(20, 5000), opa=8,
                    b=rng.choice([8, 16, 32]))
    if what == "exact":
        return dict(do="solve", kind="chain", atoms=size(20, 90), opa=4, b=4, mode="fp64", tau=0.0,
                    dirs=rng.choice([1, 3]))
    if what == "fp64":
        return dict(ladder, do="solve", kind=rng.choice(["cluster", "chain"]), atoms=size(40, 250), mode="fp64",
                    tau=rng.choice([1e-6, 1e-7]))
    if what == "fp32":
        return dict(ladder, do="solve", kind="cluster", atoms=size(40, 1000), mode="fp32")
    if what == "slab":
        return dict(ladder, do="solve", kind="slab", atoms=size(500, 4500))
    if what == "chain":
        return dict(ladder, do="solve", kind="chain", atoms=size(100, 8000))
    if what == "batch":
        lo = rng.randrange(60, 301)
        return dict(ladder, do="solve", kind="batch", atoms=lo, atoms_to=size(lo, 1000), systems=rng.randrange(2, 7))
    if what == "atom blocks":
        return dict(ladder, do="solve", kind="cluster", atoms=size(40, 1000), b=8, block_size=rng.choice([16, 32]))
    if what == "blocks":
        return dict(ladder, do="solve", kind=rng.choice(["cluster", "chain"]), atoms=size(40, 800),
                    b=rng.choice([16, 64]))
    if what == "overlap":
        return dict(ladder, do="solve", kind="cluster", atoms=size(30, 150), tau=1e-6, overlap=True)
    if what == "correct":
        return dict(ladder, do="solve", kind="cluster", atoms=size(40, 250), tau=1e-6, correct=True)
    return dict(ladder, do="solve", kind="cluster", atoms=size(40, 2000))


# ---- inputs -----------------------------------------------------------------


class Matrix:
    """A block-sparse matrix on the GPU, as the library takes it."""

    def __init__(self, nb, b, n, row_ptr, col_idx, vals):
        self.nb, self.b, self.n, self.row_ptr, self.col_idx, self.vals = nb, b, n, row_ptr, col_idx, vals

    def dense(self):
        rows = torch.repeat_interleave(torch.arange(self.nb, device=self.vals.device), self.row_ptr.long().diff())
        a = torch.zeros(self.nb, self.b, self.nb, self.b, dtype=torch.float64, device=self.vals.device)
        a[rows, :, self.col_idx.long(), :] = self.vals
        return a.reshape(self.nb * self.b, -1)[: self.n, : self.n]


class System:
    def __init__(self, h0, h1, n_electrons, s=None):
        self.h0, self.h1, self.n_electrons, self.s = h0, h1, n_electrons, s


def _distances2(a, b):
    return (a[:, None, :] - b[None, :, :]).square().sum(-1)


def _packed(n, box, gen):
    """n points in a box, no two closer than MIN_DIST (random sequential
    addition, a batch of candidates at a time)."""
    dev = gen.device
    box = torch.tensor(box, dtype=torch.float64, device=dev)
    got = torch.empty(0, 3, dtype=torch.float64, device=dev)
    while got.shape[0] < n:
        m = max(256, int(1.3 * (n - got.shape[0])))
        c = torch.rand(m, 3, dtype=torch.float64, device=dev, generator=gen) * box
        free = torch.ones(m, dtype=torch.bool, device=dev)
        for k in range(0, got.shape[0], 1024):
            free &= (_distances2(c, got[k:k + 1024]) >= MIN_DIST ** 2).all(1)
        c = c[free]
        near = torch.zeros(c.shape[0], dtype=torch.bool, device=dev)   # near an earlier candidate
        at = torch.arange(c.shape[0], device=dev)
        for k in range(0, c.shape[0], 1024):
            near |= ((_distances2(c, c[k:k + 1024]) < MIN_DIST ** 2) & (at[k:k + 1024][None, :] < at[:, None])).any(1)
        got = torch.cat([got, c[~near][: n - got.shape[0]]])
    return got


def _morton(pos):
    lo = pos.min(0).values
    q = ((pos - lo) / (pos.max(0).values - lo).max() * 1023).long()
    code = torch.zeros(pos.shape[0], dtype=torch.int64, device=pos.device)
    for bit in range(10):
        for axis in range(3):
            code |= ((q[:, axis] >> bit) & 1) << (3 * bit + axis)
    return torch.sort(code, stable=True).indices


def _blocks(ai, aj, ablk, n_atoms, opa, b):
    """Atom blocks (ai, aj) gathered in b x b blocks."""
    dev, n, g = ablk.device, n_atoms * opa, b // opa
    nb = -(-n // b)
    keys, at = torch.unique((ai // g) * nb + aj // g, return_inverse=True)
    vals = torch.zeros(keys.shape[0], b, b, dtype=torch.float64, device=dev)
    o = torch.arange(opa, device=dev)
    vals[at[:, None, None], ((ai % g) * opa)[:, None, None] + o[None, :, None],
         ((aj % g) * opa)[:, None, None] + o[None, None, :]] = ablk
    row_ptr = torch.searchsorted(torch.div(keys, nb, rounding_mode="floor"), torch.arange(nb + 1, device=dev))
    return Matrix(nb, b, n, row_ptr.int(), (keys % nb).int(), vals)


def _system(kind, n_atoms, opa, b, dirs, overlap, gen):
    dev = gen.device

    def normal(*shape):
        return torch.randn(*shape, dtype=torch.float64, device=dev, generator=gen)

    if kind == "chain":
        pos = torch.zeros(n_atoms, 3, dtype=torch.float64, device=dev)
        pos[:, 0] = SPACING * torch.arange(n_atoms, device=dev)
        cutoff = 8.0
    else:
        side = ((n_atoms / DENSITY) ** (1 / 3)) if kind == "cluster" else (n_atoms / (DENSITY * THICKNESS)) ** 0.5
        pos = _packed(n_atoms, [side, side, side if kind == "cluster" else THICKNESS], gen)
        pos = pos[_morton(pos)]
        cutoff = 10.0
    pos = pos - pos.mean(0)
    half = opa // 2
    diag = torch.zeros(n_atoms, opa, opa, dtype=torch.float64, device=dev)
    e = torch.rand(n_atoms, opa, dtype=torch.float64, device=dev, generator=gen)
    o = torch.arange(opa, device=dev)
    diag[:, o, o] = torch.where(o < half, -1.0 + 0.5 * e, 0.2 + 0.6 * e)
    pairs = []
    for k in range(0, n_atoms, 1024):
        near = _distances2(pos[k:k + 1024], pos) <= cutoff ** 2
        i, j = near.nonzero(as_tuple=True)
        pairs.append(torch.stack([i + k, j])[:, i + k < j])
    i, j = torch.cat(pairs, 1)
    r = (pos[i] - pos[j]).norm(dim=1)[:, None, None]
    atoms = torch.arange(n_atoms, device=dev)
    ai, aj = torch.cat([atoms, i, j]), torch.cat([atoms, j, i])
    hop = normal(i.shape[0], opa, opa) * (0.05 * torch.exp(-r / 1.5))
    h0 = _blocks(ai, aj, torch.cat([diag, hop, hop.transpose(1, 2)]), n_atoms, opa, b)
    h1 = []
    for d in range(dirs):
        up = torch.triu(normal(n_atoms, opa, opa) * 0.1)
        blk = up + torch.triu(up, 1).transpose(1, 2)
        blk[:, o, o] += pos[:, d, None]
        h1.append(_blocks(atoms, atoms, blk, n_atoms, opa, b))
    s = None
    if overlap:
        eye = torch.eye(opa, dtype=torch.float64, device=dev).expand(n_atoms, opa, opa)
        ovl = normal(i.shape[0], opa, opa) * (0.04 * torch.exp(-r / 2.0))
        s = _blocks(ai, aj, torch.cat([eye, ovl, ovl.transpose(1, 2)]), n_atoms, opa, b)
    return System(h0, h1, n_atoms * opa, s)


def _atoms(case):
    """(kind, atoms) of every system."""
    if case["kind"] != "batch":
        return [(case["kind"], case["atoms"])]
    lo, hi, k = case["atoms"], case["atoms_to"], case["systems"]
    return [("chain" if t % 2 else "cluster", lo + (hi - lo) * t // max(1, k - 1)) for t in range(k)]


def _systems(case, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    return [_system(kind, n, case["opa"], case["b"], case.get("dirs", 1), case.get("overlap", False), gen)
            for kind, n in _atoms(case)]


class Results:
    """Pinned host buffers for one matrix of every system, one after another,
    with room to spare: the stored blocks end where the row pointers say, and
    the rest stays zero."""

    def __init__(self, systems, blocks):
        b = systems[0].h0.b
        self.row_ptr = torch.zeros(sum(y.h0.nb + 1 for y in systems), dtype=torch.int32, pin_memory=True).numpy()
        self.reserve(blocks, b)

    def reserve(self, blocks, b):
        self.blocks = blocks
        self.col_idx = torch.zeros(blocks, dtype=torch.int32, pin_memory=True).numpy()
        self.vals = torch.zeros(blocks * b * b, dtype=torch.float64, pin_memory=True).numpy()


def _blocks_per_row(kind, n, opa, tau):
    """Stored blocks per row of 32 orbitals at threshold tau, about."""
    rows = -(-n * opa // 32)
    if tau == 0:
        return rows
    digits = -math.log10(tau)
    if kind == "chain":
        return min(rows, 1.5 * digits)
    return min(rows, rows * 24.0 * digits / (1.2 * rows + 24.0 * digits))


def prepare(case, seed):
    from paper_2009_03551_gb300 import rdm

    systems = _systems(case, seed)
    if case["do"] == "dot":
        y = systems[0]
        return dict(case=case, rdm=rdm, a=y.h0, b=y.h1[0], out=torch.empty(1, dtype=torch.float64, device="cuda"))
    solver = rdm.Solver(0)
    solver.set_params(mode=case["mode"], tau=case["tau"], tau_refine=case.get("tau_refine", -1.0),
                      tol=1e-12 if case["tau"] == 0 else 1e-9, max_iter=100, block_size=case.get("block_size", 0),
                      correct=1 if case.get("correct") else 0)
    blocks, tau = 16, min(case["tau"], case.get("tau_refine", 1.0))
    for kind, n in _atoms(case):
        rows = -(-n * case["opa"] // 32)
        blocks += int(rows * min(rows, 1.75 * _blocks_per_row(kind, n, case["opa"], tau))) * max(1, (32 // case["b"]) ** 2)
    return dict(case=case, rdm=rdm, solver=solver, systems=systems,
                results=[Results(systems, blocks) for _ in range(1 + case["dirs"])])


# ---- the pass ---------------------------------------------------------------


def run(state):
    if state["case"]["do"] == "dot":
        state["rdm"].rdm_bsr_dot_noalloc(state["a"], state["b"], state["out"].data_ptr(),
                                         torch.cuda.current_stream().cuda_stream)
        return state["out"]
    rdm, solver, systems = state["rdm"], state["solver"], state["systems"]
    solver.load(systems)
    solver.solve()
    out = {"alpha": [solver.alpha(s)[: len(y.h1), : len(y.h1)] for s, y in enumerate(systems)]}
    b = systems[0].h0.b
    for m, buf in enumerate(state["results"]):
        need = sum(rdm.rdm_get_p0_nnzb(solver.h, s) if m == 0 else rdm.rdm_get_p1_nnzb(solver.h, s, m - 1)
                   for s in range(len(systems)))
        if need > buf.blocks:
            buf.reserve(need, b)
        r = k = 0
        for s in range(len(systems)):
            view = (buf.row_ptr[r:], buf.col_idx[k:], buf.vals[k * b * b:])
            got = solver.p0(s, out=view) if m == 0 else solver.p1(s, m - 1, out=view)
            r, k = r + got.nb + 1, k + got.nnzb
        out["p1_" + "xyz"[m - 1] if m else "p0"] = {"row_ptr": buf.row_ptr, "col_idx": buf.col_idx, "vals": buf.vals}
    return out


# ---- what a pass cannot do without, and its exact results -----------------------


def work(case):
    """Inputs read and results written once; multiply-adds of the products of
    16 updates (upper triangles only: half of X0 X0 and one product for each
    X1), from an estimate of the stored blocks per row."""
    nd, size, flops = case.get("dirs", 1), 0.0, 0.0
    for kind, n in _atoms(case):
        rows = -(-n * case["opa"] // 32)
        h0 = rows * min(rows, 3.0 if kind == "chain" else 24.0) * 8192.0
        if case["do"] == "dot":
            size += 2 * rows * 8192.0
            flops += 2.0 * rows * 1024
            continue
        m = _blocks_per_row(kind, n, case["opa"], case["tau"])
        size += h0 + nd * rows * 8192.0 + (1 + nd) * rows * m * 8192.0
        flops += 16 * (0.5 + nd) * rows * m * m * 2.0 * 32 ** 3
    return {"bytes": size, "flops": flops}


def exact(case, seed):
    """Sum over states from the eigenvectors of H0: the polarizability, and
    P0 and P1 where nothing is truncated (every block is then stored)."""
    if sum(n for _, n in _atoms(case)) > 700 and case["do"] == "solve":
        return None
    systems = _systems(case, seed)
    if case["do"] == "dot":
        # over the blocks stored in both; both are zero elsewhere
        return (systems[0].h0.dense() * systems[0].h1[0].dense()).sum().reshape(1) if case["atoms"] <= 1500 else None
    alphas, mats = [], [[] for _ in range(1 + case["dirs"])]
    for y in systems:
        h0, h1 = y.h0.dense(), [h.dense() for h in y.h1]
        z = None
        if y.s is not None:
            w, v = torch.linalg.eigh(y.s.dense())
            z = (v * w.rsqrt()) @ v.T
        e, c = torch.linalg.eigh(h0 if z is None else z @ h0 @ z)
        c = c if z is None else z @ c
        k = y.n_electrons // 2
        occ, vir = c[:, :k], c[:, k:]
        ps = [occ @ occ.T]
        for h in h1:
            u = (vir.T @ h @ occ) / (e[:k][None, :] - e[k:][:, None])
            p = vir @ u @ occ.T
            ps.append(p + p.T)
        alphas.append(torch.stack([torch.stack([-2.0 * (p * h).sum() for p in ps[1:]]) for h in h1]))
        for t, p in enumerate(ps):
            nb, b = y.h0.nb, y.h0.b
            full = torch.zeros(nb * b, nb * b, dtype=torch.float64, device=p.device)
            full[: p.shape[0], : p.shape[0]] = p
            mats[t].append(full.reshape(nb, b, nb, b).transpose(1, 2).reshape(-1))
    out = {"alpha": alphas}
    for t, m in enumerate(mats):
        out["p1_" + "xyz"[t - 1] if t else "p0"] = {"row_ptr": None, "col_idx": None,
                                                    "vals": torch.cat(m) if case["tau"] == 0 else None}
    return out

"""Performance cases: what users of the solver library have it do, with sizes and inputs.

Every case goes through the public binding (paper_1605_01522_gb300.mfs) as a user's program does:
a handle is set up once for a matrix and then serves matvecs, preconditioner applications and
solves for new right-hand sides, alone or many systems at a time; one kind of case brings a new
matrix with every call and so includes the setup.  The systems are the repository's synthetic
stand-ins (inputs.py): the 2D thermo-elastic system, the 2- and 3-field 3D boxes and the split
(fluid / structure) saddle box.
"""
from functools import lru_cache
import math

import numpy as np
import torch

from paper_1605_01522_gb300 import inputs, mfs

TOL = 1e-8

# Per family: dofs per node of each field, blocks per row of a node's stencil, space dimension.
FAMILIES = {
    "te2d": dict(b=(2, 1), stencil=9, dim=2),
    "box2": dict(b=(3, 1), stencil=27, dim=3),
    "box3": dict(b=(3, 1, 1), stencil=27, dim=3),
    "split": dict(b=(3, 3, 3, 1), stencil=27, dim=3),
}
# FGMRES iterations to TOL of a mid-size member of the family (for work() only)
ITERS = {"te2d": 19, "box2": 28, "box3": 36, "split": 110}


def listed():
    return [
        # the smallest call: one coupled matvec of a small 2D system, a user's own Krylov loop
        dict(name="matvec-te2d-32", call="matvec", family="te2d", ne=32, precond="bgs_amg", precision="fp64"),
        # the coupled matvec of the 1.37 M-dof box
        dict(name="matvec-box3-64", call="matvec", family="box3", ne=64, precond="bgs_amg", precision="fp64"),
        # one float64 preconditioner application on an odd mid-size mesh, inside a user's own Krylov loop
        dict(name="apply-box3-33", call="apply", family="box3", ne=33, precond="amg_bgs", precision="fp64"),
        # the small 2D system in float64: every step of an iteration is a few microseconds
        dict(name="solve-te2d-32-fp64", call="solve", family="te2d", ne=32, precond="bgs_amg", precision="fp64"),
        # an ordinary single solve with the float32 preconditioner, monolithic AMG(BGS), odd mesh
        dict(name="solve-box3-23-amgbgs", call="solve", family="box3", ne=23, precond="amg_bgs", precision="fp32p"),
        # an ordinary single solve with SIMPLE(AMG)
        dict(name="solve-box3-40-simple", call="solve", family="box3", ne=40, precond="simple", precision="fp32p"),
        # the largest and headline solve: 1.37 M dofs, BGS(AMG), float32 preconditioner
        dict(name="solve-box3-64-fp32p", call="solve", family="box3", ne=64, precond="bgs_amg", precision="fp32p"),
        # the plain float64 arm of the box
        dict(name="solve-box3-36-fp64", call="solve", family="box3", ne=36, precond="bgs_amg", precision="fp64"),
        # the saddle system of the split box, float64 (four fields, blocks of different patterns)
        dict(name="solve-split-20-simple", call="solve", family="split", ne=20, precond="simple", precision="fp64"),
        # many different systems solved together (log-uniform sizes)
        dict(name="batch-box2-24", call="batch", family="box2", ne=24, nsys=24, precond="bgs_amg",
             precision="fp32p"),
        # one matrix, many right-hand sides solved together
        dict(name="batch-te2d-32x96", call="clones", family="te2d", ne=32, nsys=96, precond="bgs_amg",
             precision="fp64"),
        # a request of a server that brings its own matrix: setup, solve from host buffers, free
        dict(name="new-box3-21", call="new", family="box3", ne=21, precond="bgs_amg", precision="fp32p"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges, none of the listed ones."""
    known = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        case = _draw(rng)
        if case not in known:
            return case


def _draw(rng):
    call = rng.choice(["matvec", "apply", "solve", "solve", "solve", "batch", "clones", "new"])
    if call in ("matvec", "apply"):
        family = rng.choice(["te2d", "box2", "box3"] + (["split"] if call == "matvec" else []))
        ne = {"te2d": _log_uniform(rng, 9, 200), "split": _log_uniform(rng, 7, 28)}.get(family)
        ne = ne or _log_uniform(rng, 6, 50)
        if call == "matvec":
            return dict(call=call, family=family, ne=ne, precond="simple" if family == "split" else "bgs_amg",
                        precision="fp64")
        return dict(call=call, family=family, ne=ne, precond=rng.choice(["bgs_amg", "amg_bgs", "simple"]),
                    precision="fp64")
    if call == "solve":
        family = rng.choice(["te2d", "te2d", "box2", "box3", "box3", "split"])
        if family == "split":
            return dict(call=call, family=family, ne=_log_uniform(rng, 7, 24), precond="simple",
                        precision="fp64")
        ne = _log_uniform(rng, 9, 160) if family == "te2d" else _log_uniform(rng, 7, 50)
        return dict(call=call, family=family, ne=ne, precond=rng.choice(["bgs_amg", "bgs_amg", "amg_bgs", "simple"]),
                    precision=rng.choice(["fp32p", "fp32p", "fp64"]))
    if call == "batch":
        return dict(call=call, family="box2", ne=_log_uniform(rng, 14, 26), nsys=rng.randint(3, 24),
                    precond="bgs_amg", precision="fp32p")
    if call == "clones":
        return dict(call=call, family="te2d", ne=_log_uniform(rng, 9, 40), nsys=_log_uniform(rng, 4, 128),
                    precond=rng.choice(["bgs_amg", "amg_bgs"]), precision=rng.choice(["fp32p", "fp64"]))
    return dict(call=call, family=rng.choice(["box2", "box3"]), ne=_log_uniform(rng, 8, 26),
                precond=rng.choice(["bgs_amg", "simple"]), precision="fp32p")


def _assemble(family, ne, seed):
    if family == "te2d":
        return inputs.thermo_elastic_2d(ne=ne)
    if family == "split":
        return inputs.fsi_box(ne=ne)
    return inputs.coupled_box_3d(ne=ne, nfields=3 if family == "box3" else 2, seed=seed)


# A program that keeps a handle keeps one matrix: it depends on the family and the size alone.
_system = lru_cache(maxsize=48)(lambda family, ne: _assemble(family, ne, 1))


def _rhs(system, seed):
    """N(0, 1) right-hand side, zero on the Dirichlet nodes of each field."""
    b = np.random.default_rng(seed).standard_normal(system.ndofs)
    for off, f in zip(system.offsets, system.fields):
        b[off:off + f.ndofs].reshape(f.nnodes, f.b)[f.dirichlet_nodes] = 0.0
    return b


def _batch_sizes(case):
    """Mesh edges of a batch, log-uniform up to case["ne"]; fixed by the case."""
    rng = np.random.default_rng(case["nsys"])
    return [int(v) for v in np.rint(np.exp(rng.uniform(math.log(8), math.log(case["ne"]), case["nsys"])))]


def _params(case):
    # levels as the repository's benchmark takes them for these systems
    levels = dict(max_levels=3, coarse_max=0) if case["family"] == "te2d" else dict(max_levels=5, coarse_max=1000)
    kw = dict(precond=case["precond"], precision=case["precision"], **levels)
    if case["family"] == "split":
        kw.update(simple_group=[0, 0, 0, 1], simple_approx="diag")
    if case["call"] in ("batch", "clones"):
        kw["layout_tune"] = 1
    return kw


def _host_inputs(case, seed):
    """(systems, right-hand sides) of a case on the host."""
    if case["call"] == "new":
        s = _assemble(case["family"], case["ne"], seed)
        return [s], [_rhs(s, seed)]
    if case["call"] == "batch":
        systems = [_system(case["family"], ne) for ne in _batch_sizes(case)]
        return systems, [_rhs(s, 1000 * seed + k) for k, s in enumerate(systems)]
    s = _system(case["family"], case["ne"])
    n = case["nsys"] if case["call"] == "clones" else 1
    return [s], [_rhs(s, 1000 * seed + k) for k in range(n)]


def prepare(case, seed):
    systems, rhs = _host_inputs(case, seed)
    state = dict(call=case["call"], rhs=rhs)
    if case["call"] == "new":
        state.update(system=systems[0], kw=_params(case))
        return state
    solvers = [mfs.Solver(s, **_params(case)) for s in systems]
    if case["call"] == "clones":
        solvers += [solvers[0].clone() for _ in range(case["nsys"] - 1)]
    state.update(solvers=solvers, rhs=[torch.from_numpy(b).cuda() for b in rhs])
    return state


def run(state):
    call = state["call"]
    if call == "matvec":
        return state["solvers"][0].matvec(state["rhs"][0])
    if call == "apply":
        return state["solvers"][0].apply(state["rhs"][0])
    if call == "solve":
        x, info, _ = state["solvers"][0].solve(state["rhs"][0], tol=TOL)
        return dict(x=x, iters=info["iters"])
    if call in ("batch", "clones"):
        xs, infos, _ = mfs.solve_batch(state["solvers"], state["rhs"], tol=TOL)
        x = torch.cat(xs)
        return dict(x=x, iters=np.array([i["iters"] for i in infos]))
    with mfs.Solver(state["system"], **state["kw"]) as solver:
        x, info, _ = solver.solve(state["rhs"][0], tol=TOL)
    return dict(x=x, iters=info["iters"])


def _shape(family, ne):
    """(dofs, entries, blocks) of the coupled matrix and (entries, blocks) of its diagonal blocks."""
    f = FAMILIES[family]
    if family == "split":
        nodes = (ne + 1) ** 2 * (ne // 2 + 1)
        pairs = [(0, 0), (1, 1), (2, 2), (3, 3), (2, 3), (3, 2), (2, 1)]
    else:
        nodes = (ne + 1) ** f["dim"]
        pairs = [(i, j) for i in range(len(f["b"])) for j in range(len(f["b"]))]
    node_pairs = (3 * ne + 1) ** f["dim"] if family != "split" else (3 * ne + 1) ** 2 * (3 * (ne // 2) + 1)
    entries = sum(node_pairs * f["b"][i] * f["b"][j] for i, j in pairs)
    diag = sum(node_pairs * b * b for b in f["b"])
    return nodes * sum(f["b"]), entries, node_pairs * len(pairs), diag, node_pairs * len(f["b"])


def _iteration_work(case, ne):
    """Bytes and flops of one FGMRES iteration (mid-cycle basis of half the iterations) and n."""
    n, ent, blk, dent, dblk = _shape(case["family"], ne)
    s = 4 if case["precision"] == "fp32p" else 8
    k = min(50, ITERS[case["family"]]) / 2
    a_bytes, a_flops = _apply_work(case, ne)
    m_bytes, m_flops = 8 * ent + 4 * blk + 16 * n, 2 * ent
    basis = 3 * 8 * n * k + 6 * 8 * n  # h1, then w and h2, then w again
    return a_bytes + m_bytes + basis + (2 * s + 16) * n, a_flops + m_flops + 8 * n * k, n


def _apply_work(case, ne):
    """One application: on every level two pre-, one residual and two post-smoothing passes, the
    first from zero (so four matrix passes), and one pass over half the coupling blocks; the coarse
    levels and transfers add about a third of the finest level's matrix."""
    n, ent, blk, dent, dblk = _shape(case["family"], ne)
    s = 4 if case["precision"] == "fp32p" else 8
    diag = s * dent + 4 * dblk
    coup = 0.5 * (s * (ent - dent) + 4 * (blk - dblk))
    return 4.33 * diag + coup + 12 * s * n, 2 * (4.33 * dent + 0.5 * (ent - dent)) + 12 * n


def work(case):
    if case["call"] == "matvec":
        n, ent, blk, _, _ = _shape(case["family"], case["ne"])
        return dict(bytes=8 * ent + 4 * blk + 16 * n, flops=2 * ent)
    if case["call"] == "apply":
        b, f = _apply_work(case, case["ne"])
        return dict(bytes=b, flops=f)
    sizes = _batch_sizes(case) if case["call"] == "batch" else [case["ne"]] * case.get("nsys", 1)
    it = ITERS[case["family"]]
    total = [_iteration_work(case, ne) for ne in sizes]
    b = it * sum(t[0] for t in total)
    if case["call"] == "new":  # the input blocks are read, and written in the layouts that are kept
        _, ent, blk, _, _ = _shape(case["family"], case["ne"])
        b += 2 * (8 * ent + 4 * blk)
    return dict(bytes=b, flops=it * sum(t[1] for t in total))


def _dense(system):
    n, off = system.ndofs, system.offsets
    A = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    for (i, j), m in system.blocks.items():
        rows = torch.from_numpy(np.repeat(np.arange(m.nbrows), np.diff(m.rowptr))).cuda()
        cols = torch.from_numpy(m.colind.astype(np.int64)).cuda()
        vals = torch.from_numpy(m.vals).cuda()
        for r in range(m.br):
            for c in range(m.bc):
                A[off[i] + rows * m.br + r, off[j] + cols * m.bc + c] = vals[:, r, c]
    return A


def _product(system, x):
    """A x in float64 by plain torch, block by block."""
    off = system.offsets
    y = torch.zeros_like(x)
    for (i, j), m in system.blocks.items():
        xj = x[off[j]:off[j + 1]].reshape(-1, m.bc)
        cols = torch.from_numpy(m.colind.astype(np.int64)).cuda()
        rows = torch.from_numpy(np.repeat(np.arange(m.nbrows), np.diff(m.rowptr))).cuda()
        prod = torch.einsum("krc,kc->kr", torch.from_numpy(m.vals).cuda(), xj[cols])
        y[off[i]:off[i + 1]].reshape(-1, m.br).index_add_(0, rows, prod)
    return y


def exact(case, seed):
    """Products by plain torch; solutions by a dense solve where the system is small enough.  A
    preconditioner application has no value of its own apart from its hierarchy."""
    if case["call"] == "apply":
        return None
    if case["call"] != "matvec" and (case["call"] == "batch" or _shape(case["family"], case["ne"])[0] > 9000):
        return None
    systems, rhs = _host_inputs(case, seed)
    if case["call"] == "matvec":
        return _product(systems[0], torch.from_numpy(rhs[0]).cuda())
    b = torch.from_numpy(np.stack(rhs, axis=1)).cuda()
    x = torch.linalg.solve(_dense(systems[0]), b)
    return dict(x=x.T.reshape(-1), iters=None)

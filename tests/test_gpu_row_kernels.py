"""Row layouts, fused V-cycle steps, CGS2 passes and the block SpGEMM at the
sizes where their dispatch changes.  Needs a GB300.

Applications are compared with the FP64 oracle on the library's exported
hierarchy within the 1e-12 (relative, max-norm) of the other parity tests:
float64 kernels and oracle differ only in the order of their sums.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1605_01522_gb300 import inputs, mfs
from tests.oracle_from_lib import oracle_preconditioner

pytestmark = pytest.mark.gpu


def _system(name):
    kind, ne = name.split("-")
    if kind == "te2d":
        return inputs.thermo_elastic_2d(ne=int(ne)), dict(max_levels=3, coarse_max=0)
    if kind == "split":
        return inputs.fsi_box(ne=int(ne)), dict(max_levels=3, coarse_max=100)
    return inputs.coupled_box_3d(ne=int(ne), nfields=int(kind[-1])), dict(max_levels=4, coarse_max=150)


# rows of the fine fields: 676 / 729 (plain BSR; SELL-32 from 700 on in batch setups), 8,281 and 9,261
# (short rows SELL-32, the others plain BSR), 17,576 (SELL-32, 549.25 slices); products of one field
# (box2), two (box3) and three (split) terms; kernel: a layout that has to be among the launches
@pytest.mark.parametrize("name,pc,tune,kernel", [
    ("te2d-25", "bgs_amg", 1, "smooth_warp"),
    ("box3-8", "amg_bgs", 0, "terms_bsr"),
    ("box3-8", "amg_bgs", 1, "sell_split"),
    ("te2d-90", "amg_bgs", 0, "sell_split"),
    ("box2-20", "simple", 0, "terms_bsr"),
    ("box3-25", "amg_bgs", 0, "terms_sell"),
    ("box2-25", "simple", 0, "terms_sell"),
    ("split-9", "simple", 0, "terms_bsr"),
])
def test_application_matches_oracle_at_layout_edges(name, pc, tune, kernel):
    s, kw = _system(name)
    with mfs.Solver(s, precond=pc, layout_tune=tune, profile=1, max_iters=2, **kw) as lib:
        v = np.random.default_rng(3).standard_normal(s.ndofs)
        z = lib.apply(torch.from_numpy(v).cuda()).cpu().numpy()
        zr = oracle_preconditioner(lib, s)(v)
        assert np.abs(z - zr).max() <= 1e-12 * np.abs(zr).max()
        lib.solve(torch.from_numpy(s.rhs).cuda(), tol=1e-8)
        assert any(kernel in r[0] for r in lib.kernel_detail())


@pytest.mark.parametrize("order,sweeps", [("sym", 1), ("fwd", 2)])
@pytest.mark.parametrize("pc", ["bgs_amg", "amg_bgs", "amg_simple"])
def test_fused_steps_with_second_visits(pc, order, sweeps):
    """A field that is visited again (symmetric order, second sweep) starts
    from a nonzero vector: its couplings include its own block."""
    s, kw = _system("box3-6")
    with mfs.Solver(s, precond=pc, bgs_order=order, bgs_sweeps=sweeps, **kw) as lib:
        v = np.random.default_rng(4).standard_normal(s.ndofs)
        z = lib.apply(torch.from_numpy(v).cuda()).cpu().numpy()
        zr = oracle_preconditioner(lib, s)(v)
        assert np.abs(z - zr).max() <= 1e-12 * np.abs(zr).max()


@pytest.mark.parametrize("n", [1, 31, 255, 256, 257, 152 * 256 - 1, 152 * 256 + 1, 2 * 152 * 256 + 1,
                               608 * 256 + 1, 1000003])
def test_dot_at_tile_edges(n):
    """One 256-entry tile, the next CTA, the next CTA per SM, several tiles
    per CTA.  Bound: 1e-13 of the sum of the products' magnitudes, far above
    the n / 256 / 32 + 30 roundings of a sum in chains and trees."""
    rng = np.random.default_rng(n)
    x, y = rng.standard_normal(n), rng.standard_normal(n)
    d = mfs.dot_noalloc(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    assert abs(d - float(np.dot(x, y))) <= 1e-13 * float(np.abs(x) @ np.abs(y))


def test_dot_with_the_most_partial_sums_then_fewer():
    """194,560 entries are 760 tiles of 256, one CTA each: the largest number of
    partial sums of any length.  A shorter call afterwards reads only its own."""
    rng = np.random.default_rng(11)
    for n in (194560, 194559, 194560 - 256 + 3, 5037, 194560, 77):
        x, y = rng.standard_normal(n), rng.standard_normal(n)
        xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
        d = mfs.dot_noalloc(xd, yd)
        assert abs(d - float(np.dot(x, y))) <= 1e-13 * float(np.abs(x) @ np.abs(y))
        assert d == mfs.dot_noalloc(xd, yd)


@pytest.mark.parametrize("restart", [5, 33, 60])
@pytest.mark.parametrize("tune", [0, 1])
def test_basis_stays_orthogonal_at_every_row_count(restart, tune):
    """The residual estimate of the Givens recurrence equals the true
    residual as long as the basis is orthonormal: with a twice-orthogonalised
    basis to rounding (kappa eps of the operator is below 1e-10 here), for
    cycles shorter than a warp's rows, past 32 rows and up to the longest."""
    s, kw = _system("split-9")
    with mfs.Solver(s, precond="simple", restart=restart, max_iters=min(3 * restart, 60), layout_tune=tune, **kw) as lib:
        _, info, _ = lib.solve(torch.from_numpy(s.rhs).cuda(), tol=1e-12)
        assert abs(info["est_relres"] - info["true_relres"]) <= 1e-6 * info["true_relres"] + 1e-14


@pytest.mark.parametrize("pc,kw", [
    ("simple", dict(simple_group=[1, 0, 0])),   # S~ of 3x3 blocks, 125 columns a row: past the shared accumulators
    ("bgs_amg", dict()),                        # 6x6 Galerkin rows in them
])
def test_device_products_equal_host_products(pc, kw):
    s, base = _system("box3-7")
    g = mfs.Solver(s, precond=pc, setup_device=1, **base, **kw)
    h = mfs.Solver(s, precond=pc, setup_device=0, **base, **kw)
    groups = [(0, 2 if pc == "simple" else 3)] + ([(1, 1)] if pc == "simple" else [])
    for grp, nf in groups:
        for lev in range(g.num_levels(grp)):
            for i in range(nf):
                A, B = g.export_csr("A", grp, lev, i, i), h.export_csr("A", grp, lev, i, i)
                assert (A.indptr == B.indptr).all() and (A.indices == B.indices).all()
                assert np.abs(A.data - B.data).max() <= 1e-12 * np.abs(B.data).max()
    g.close()
    h.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32p"])
@pytest.mark.parametrize("name,pc", [("box3-25", "amg_bgs"), ("box2-25", "simple"), ("box2-50", "bgs_amg")])
def test_programmatic_launches_equal_ordinary_ones_on_split_sell(name, pc, prec):
    """17,576 and 132,651 rows: the SELL-32 kernels with several threads a row
    (alone and as fused products) and with one thread a row run as programmatic
    dependent launches and still read their predecessors' results."""
    s, kw = _system(name)
    v = torch.from_numpy(np.random.default_rng(8).standard_normal(s.ndofs)).cuda()
    b = torch.from_numpy(s.rhs).cuda()
    with mfs.Solver(s, precond=pc, precision=prec, pdl=0, **kw) as off:
        z, y = off.apply(v), off.matvec(v)
        x, info, _ = off.solve(b, tol=1e-8)
        for pdl in (1, -1):
            with mfs.Solver(s, precond=pc, precision=prec, pdl=pdl, **kw) as on:
                for _ in range(3):
                    assert torch.equal(z, on.apply(v)) and torch.equal(y, on.matvec(v))
                xp, ip, _ = on.solve(b, tol=1e-8)
                assert ip["iters"] == info["iters"] and torch.equal(x, xp)

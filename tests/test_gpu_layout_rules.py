"""Which row kernel the layout rules give a matrix, and its product against
scipy, for matrices that no mesh of the repository has.  Needs a GB300.

The handle takes the single-level Gauss-Seidel preconditioner (no hierarchy), so that
any square matrix with a full diagonal can be given; a profiled solve names the
kernels of the float64 products.  Bound of an entry of a product: (k + 64)
2^-53 of |A| |x| with k terms in the longest row, what scipy's one chain may be
off by (the kernels' shorter chains and the sums over lanes are off by less).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import scipy.sparse as sp

from paper_1605_01522_gb300 import inputs, mfs
from tests.oracle_from_lib import oracle_preconditioner

pytestmark = pytest.mark.gpu


def _banded(n, width, b, long_rows=0, length=0, seed=0):
    """n block rows of `width` blocks around the diagonal (fewer at the ends),
    `long_rows` of them with about `length` random columns more."""
    rng = np.random.default_rng(seed)
    off = np.arange(width) - width // 2
    r = np.repeat(np.arange(n), width)
    c = r + np.tile(off, n)
    keep = (c >= 0) & (c < n)
    r, c = r[keep], c[keep]
    for k in range(long_rows):
        row = (k * n) // max(1, long_rows) + 5
        r = np.concatenate([r, np.full(length, row)])
        c = np.concatenate([c, rng.choice(n, length, replace=False)])
    key = np.unique(r.astype(np.int64) * n + c)
    r, c = key // n, key % n
    rp = np.searchsorted(r, np.arange(n + 1)).astype(np.int32)
    v = rng.uniform(-1.0, 1.0, (len(r), b, b))
    v[r == c] += 8.0 * np.eye(b)
    return inputs.BSR(b, b, n, n, rp, c.astype(np.int32), v)


def _system(m):
    n = m.nbrows
    f = inputs.Field("u", m.br, n, 3, np.zeros((n, 3)), "const")
    rhs = np.random.default_rng(1).standard_normal(n * m.br)
    return inputs.BlockSystem([f], {(0, 0): m}, rhs, name="banded")


def _check(s, kernels, **kw):
    """kernels: names that have to be among the solve's, or with a leading '-' must not be"""
    A = sp.bmat([[s.blocks[(i, j)].to_scipy() if (i, j) in s.blocks else None for j in range(s.nfields)]
                 for i in range(s.nfields)]).tocsr()
    x = np.random.default_rng(2).standard_normal(s.ndofs)
    with mfs.Solver(s, precond="bgs_gs", smoother="gs", profile=1, max_iters=2, **kw) as lib:
        y = lib.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
        bound = (np.diff(A.indptr).max() + 64) * 2.0 ** -53
        assert (np.abs(y - A @ x) <= bound * (abs(A) @ abs(x))).all()
        lib.solve(torch.from_numpy(s.rhs).cuda(), tol=1e-8, check=False)
        names = [r[0] for r in lib.kernel_detail()]
    for k in kernels.split():
        assert any(k.lstrip("-") in n for n in names) != k.startswith("-"), (k, names)


@pytest.mark.parametrize("n,b,long_rows,length,tune,kernels", [
    (20001, 1, 0, 0, 0, "spmv_sell_split<1x1,f64>"),            # even rows: SELL-32
    (20001, 1, 3, 200, 0, "spmv_sell_split<1x1,f64>"),          # 200 blocks of one entry: still
    (20001, 1, 3, 300, 0, "spmv_warp<1x1,f64> -sell_split"),    # 300: plain BSR
    (20001, 3, 1, 60, 0, "spmv_warp<3x3,f64> -sell_split"),     # 3x3 blocks: from 57 on
    (20001, 1, 2, 4000, 0, "spmv_warp<1x1,f64> -sell_split"),   # all 32 lanes
    (1000, 2, 0, 0, 1, "spmv_sell_split<2x2,f64>"),             # batch setups
    (1000, 2, 2, 300, 1, "spmv_warp<2x2,f64> -sell_split"),
])
def test_few_long_rows_keep_plain_bsr(n, b, long_rows, length, tune, kernels):
    """The threads of a SELL-32 row walk it alone: one row of 4,000 3x3 blocks
    among 68,921 of 27 took 3 ms there, 0.2 ms over the lanes of plain BSR."""
    _check(_system(_banded(n, 27, b, long_rows, length)), kernels, layout_tune=tune)


@pytest.mark.parametrize("n,tune,kernels", [
    (16383, 0, "spmv_warp<6x6,f64> -sell"),
    (16384, 0, "spmv_sell_split<6x6,f64>"),
    (701, 1, "spmv_sell_split<6x6,f64>"),
])
def test_blocks_of_six_dofs_follow_the_rows(n, tune, kernels):
    """Fine fields with six dofs a node (68,921 rows: 198 us as plain BSR, 142)."""
    _check(_system(_banded(n, 27, 6)), kernels, layout_tune=tune)


@pytest.mark.parametrize("rows,length,b,kernels", [
    (4, 767, 3, "spmv_warp<1x3,f64>"),            # constraint rows: a warp each
    (4, 768, 3, "spmv_cta<1x3,f64>"),             # a CTA each
    (1024, 800, 1, "spmv_cta<1x1,f64>"),
    (1025, 800, 1, "spmv_warp<1x1,f64>"),
    (3, 5000, 6, "spmv_cta<1x6,f64>"),
])
def test_few_very_long_rows_take_a_cta_each(rows, length, b, kernels):
    """Rows of multipliers against a large field; a warp walked 20 rows of
    3,000 1x1 blocks in 46 us, a CTA a row in 35."""
    n = 6000
    rng = np.random.default_rng(3)
    big = _banded(n, 9, b)
    ci = np.concatenate([np.sort(rng.choice(n, length, replace=False)) for _ in range(rows)]).astype(np.int32)
    A10 = inputs.BSR(1, b, rows, n, (np.arange(rows + 1) * length).astype(np.int32), ci,
                     rng.uniform(-1.0, 1.0, (rows * length, 1, b)))
    one = np.arange(rows + 1, dtype=np.int32)
    A11 = inputs.BSR(1, 1, rows, rows, one, one[:-1].copy(), np.ones((rows, 1, 1)))
    s = _system(big)
    s.fields.append(inputs.Field("c", 1, rows, 3, np.zeros((rows, 3)), "const"))
    s.blocks.update({(1, 0): A10, (1, 1): A11})
    s.rhs = np.concatenate([s.rhs, np.ones(rows)])
    # one product a row field would hide the kernel's name in a fused launch: batch setups keep them apart
    _check(s, kernels, layout_tune=1)


@pytest.mark.parametrize("fields,n,width,same_as_four", [
    ((3, 1, 1), 2, 2, True),
    ((3, 1, 1), 33, 27, False),     # 8 threads a row; rows of one block, of 14 and of 27
    ((3, 1), 2047, 27, False),
    ((2, 1), 2500, 20, False),
    ((2, 1), 2501, 20, True),
    ((3, 1, 1), 1000, 12, True),    # short rows
])
def test_merged_rows_take_the_threads_of_the_rule(fields, n, width, same_as_four):
    """The coupled matvec without rows_split, whose order of sums (and so its
    bits) is the one with 4 threads a row or, for few long rows, with 8."""
    rng = np.random.default_rng(n)
    base = _banded(n, width, 1)
    row = np.repeat(np.arange(n), np.diff(base.rowptr))
    keep = (row % 13 != 12) | (base.colind == row)  # every 13th row: its diagonal alone
    rp = np.searchsorted(row[keep], np.arange(n + 1)).astype(np.int32)
    ci = base.colind[keep]
    s = inputs.BlockSystem([], {}, rng.standard_normal(n * sum(fields)), name="banded")
    for i, b in enumerate(fields):
        s.fields.append(inputs.Field(f"f{i}", b, n, 3, np.zeros((n, 3)), "const"))
        for j, c in enumerate(fields):
            v = rng.uniform(-1.0, 1.0, (len(ci), b, c))
            if i == j:
                v[row[keep] == ci] += 8.0 * np.eye(b)
            s.blocks[(i, j)] = inputs.BSR(b, c, n, n, rp, ci, v)
    _check(s, "spmv_rows")
    x = torch.from_numpy(rng.standard_normal(s.ndofs)).cuda()
    kw = dict(precond="bgs_gs", smoother="gs")
    with mfs.Solver(s, **kw) as a, mfs.Solver(s, rows_split=4, **kw) as b:
        assert torch.equal(a.matvec(x), b.matvec(x)) == same_as_four


@pytest.mark.parametrize("ne,prec,tol", [(30, "fp64", 1e-12), (33, "fp64", 1e-12), (47, "fp32p", 2e-3)])
def test_batch_setups_keep_the_vcycle_tail(ne, prec, tol):
    """Scalar levels of 700 rows and more that fit the one-CTA tail (961 and
    1,156 rows in float64, 2,304 in float32) take it in batch setups too.
    Bounds: the other application tests' for float64; in float32 a rounding of
    6e-8 from each of 16 steps, times the condition of the coarse matrices
    (1,784 for elasticity)."""
    s = inputs.thermo_elastic_2d(ne=ne)
    v = np.random.default_rng(3).standard_normal(s.ndofs)
    with mfs.Solver(s, precond="bgs_amg", precision=prec, layout_tune=1, vcycle_tail=1, profile=1, max_iters=2,
                    max_levels=2, coarse_max=0) as lib:
        z = lib.apply(torch.from_numpy(v).cuda()).cpu().numpy()
        zr = oracle_preconditioner(lib, s)(v)
        assert np.abs(z - zr).max() <= tol * np.abs(zr).max()
        lib.solve(torch.from_numpy(s.rhs).cuda(), tol=1e-8, check=False)
        assert any(r[0] == "vcycle_tail" for r in lib.kernel_detail())


def _coupled(n, width, nf, wide=None, wide_width=0):
    """nf scalar fields of n nodes, all pairs coupled; block `wide` has rows of wide_width."""
    s = inputs.BlockSystem([], {}, np.random.default_rng(4).standard_normal(n * nf), name="coupled")
    for i in range(nf):
        s.fields.append(inputs.Field(f"f{i}", 1, n, 3, np.zeros((n, 3)), "const"))
        for j in range(nf):
            s.blocks[(i, j)] = _banded(n, wide_width if (i, j) == wide else width, 1, seed=10 * i + j)
    return s


@pytest.mark.parametrize("n,width,nf,wide,wide_width,kernels", [
    (333, 9, 4, None, 0, "spmv_terms_bsr<1x4,f64>"),                             # four products: one launch
    (333, 9, 5, None, 0, "spmv_warp<1x1,f64> spmv_terms_bsr<1x4,f64>"),          # five: one by one (the sweep's four fused)
    (20001, 27, 2, None, 0, "spmv_terms_sell<1x2,f64> -spmv_warp"),
    (20001, 27, 2, (0, 1), 161, "spmv_warp<1x1,f64> spmv_sell_split<1x1,f64> spmv_terms_sell<1x2,f64>"),  # two layouts in row 0
])
def test_products_of_a_row_are_fused_where_the_layouts_allow_it(n, width, nf, wide, wide_width, kernels):
    _check(_coupled(n, width, nf, wide, wide_width), kernels)


@pytest.mark.parametrize("length,kernels", [(767, "spmv_terms_bsr<1x2,f64> -spmv_cta"), (768, "spmv_cta<1x3,f64> -terms")])
def test_cta_rows_stay_out_of_fused_products(length, kernels):
    n, rows = 6000, 5
    rng = np.random.default_rng(6)
    ci = np.concatenate([np.sort(rng.choice(n, length, replace=False)) for _ in range(rows)]).astype(np.int32)
    one = np.arange(rows + 1, dtype=np.int32)
    s = _system(_banded(n, 9, 3))
    s.fields.append(inputs.Field("c", 1, rows, 3, np.zeros((rows, 3)), "const"))
    s.blocks[(1, 0)] = inputs.BSR(1, 3, rows, n, (np.arange(rows + 1) * length).astype(np.int32), ci,
                                  rng.uniform(-1.0, 1.0, (rows * length, 1, 3)))
    s.blocks[(1, 1)] = inputs.BSR(1, 1, rows, rows, one, one[:-1].copy(), np.ones((rows, 1, 1)))
    s.rhs = np.concatenate([s.rhs, np.ones(rows)])
    _check(s, kernels, bgs_order="fwd")

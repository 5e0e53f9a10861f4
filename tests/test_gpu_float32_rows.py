"""Float32 row kernels (several threads a row, fused products, a CTA a row)
against the float64 oracle on the library's exported hierarchy.  Needs a GB300.

Couplings are strong here (alpha = beta = 20): an application without one of the
coupling blocks is 0.1 to 1.1 off in the norm of a field.  Bound, per field in
the 2-norm: 64 2^-24 times the condition (1-norm) of the coarsest matrices - the
matrix and every one of some 60 steps are rounded once, and the coarse solve
amplifies what reaches it by at most its condition; 1e-4 to 1e-3 here.  For
float64 64 + k times 2^-53 with k terms in the longest row, which the oracle adds
in one chain.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import precond
from paper_1605_01522_gb300 import inputs, mfs
from tests.oracle_from_lib import oracle_preconditioner
from tests.test_gpu_layout_rules import _banded, _system as _one_field

pytestmark = pytest.mark.gpu


def _cond(A):
    A = A.toarray() if hasattr(A, "toarray") else np.asarray(A)
    return np.linalg.norm(A, 1) * np.linalg.norm(np.linalg.inv(A), 1)


def _coarse_condition(lib, s, pc):
    c, nf = 1.0, s.nfields
    if pc == "amg_bgs":
        L = lib.num_levels(0) - 1
        blocks = {(i, j): lib.export_csr("A", 0, L, i, j) for (i, j) in s.blocks}
        return _cond(precond.assemble(blocks, nf))
    groups = [(0, range(nf - 1)), (1, range(1))] if pc == "simple" else [(0, range(nf))]
    for g, fields in groups:
        for i in fields:
            c = max(c, _cond(lib.export_csr("A", g, lib.num_levels(g) - 1, i, i)))
    return c


def _compare(s, kernels, **kw):
    prec = kw["precision"]
    v = np.random.default_rng(3).standard_normal(s.ndofs)
    with mfs.Solver(s, profile=1, max_iters=2, **kw) as lib:
        z = lib.apply(torch.from_numpy(v).cuda()).cpu().numpy()
        zr = oracle_preconditioner(lib, s)(v)
        longest = max(np.diff(b.rowptr).max() * b.bc for b in s.blocks.values())
        roundings = 64 * 2.0 ** -24 if prec == "fp32p" else (64 + longest) * 2.0 ** -53
        tol = roundings * _coarse_condition(lib, s, kw["precond"])
        for lo, hi in zip(s.offsets[:-1], s.offsets[1:]):
            assert np.linalg.norm((z - zr)[lo:hi]) <= tol * np.linalg.norm(zr[lo:hi])
        lib.solve(torch.from_numpy(s.rhs).cuda(), tol=1e-8, check=False)
        names = [r[0] for r in lib.kernel_detail()]
    for k in kernels.split():
        assert any(k in n for n in names), (k, names)


# rows: 17,576 SELL-32 with several threads, 9,261 plain BSR (P SELL-32), 1,000 in a batch setup
@pytest.mark.parametrize("ne,pc,tune,kernels", [
    (25, "amg_bgs", 0, "smooth_terms_sell<3x2,f32> spmv_terms_sell<3x2,f32> smooth_sell_split<3x3,f32>"),
    (25, "simple", 0, "spmv_terms_sell<3x1,f32> spmv_terms_sell<1x1,f32> spmv_sell_split<3x6,f32>"),
    (25, "bgs_amg", 0, "spmv_terms_sell<3x1,f32> smooth_sell_split<1x1,f32>"),
    (20, "amg_bgs", 0, "smooth_terms_bsr<3x2,f32> spmv_terms_bsr<1x2,f32> smooth_warp<3x3,f32>"),
    (9, "bgs_amg", 1, "smooth_sell_split<3x3,f32> smooth_sell_split<1x1,f32>"),
])
def test_float32_application_matches_oracle(ne, pc, tune, kernels):
    s = inputs.coupled_box_3d(ne=ne, nfields=2, alpha=20.0, beta=20.0)
    _compare(s, kernels, precond=pc, precision="fp32p", layout_tune=tune, max_levels=3, coarse_max=100)


@pytest.mark.parametrize("n,width,b,prec,kernels", [
    (4096, 161, 1, "fp32p", "smooth_cta<1x1,f32>"),     # 128 blocks a row and more, up to 4,096 rows
    (1001, 201, 3, "fp32p", "smooth_cta<3x3,f32>"),
    (1023, 2045, 1, "fp64", "smooth_cta<1x1,f64>"),     # every row full: 768 blocks and more, up to 1,024 rows
    (16384, 27, 6, "fp32p", "smooth_sell_split<6x6,f32>"),
    (16384, 27, 6, "fp64", "smooth_sell_split<6x6,f64>"),
])
def test_smoothing_steps_of_wide_rows_and_blocks(n, width, b, prec, kernels):
    m = _banded(n, width, b)
    m.vals[np.repeat(np.arange(n), np.diff(m.rowptr)) == m.colind] += 0.6 * b * width * np.eye(b)  # dominant diagonal
    _compare(_one_field(m), kernels, precond="bgs_amg", precision=prec, max_levels=3, coarse_max=10)

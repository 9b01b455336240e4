"""Kernels at the edges of their tiles, each against plain numpy on the CSR or the oracle's rule."""
import numpy as np
import pytest

import paper_1411_0660_gb300 as g


@pytest.fixture(scope="module")
def ctx():
    return g.Context(0)


@pytest.mark.gpu
@pytest.mark.parametrize("L,nup", [(5, 2), (8, 4), (11, 5), (12, 6), (13, 7)])
@pytest.mark.parametrize("prec", [g.MBL_PREC_FP32, g.MBL_PREC_FP64])
@pytest.mark.parametrize("nrhs", [1, 7, 8, 9, 32])
def test_refined_solve_leaves_a_small_residual(ctx, L, nup, prec, nrhs):
    """Every block width's padding and every narrow-panel shape: the refined solve stops at a normwise
    backward error of 1e-14, so |b - (H - s) x| <= 1e-14 (|A| |x| + |b|) per column; the residual computed
    here in another order adds rounding of at most nnz-per-row ulps, 2e-15 relative: 2e-14 in all."""
    sec = g.build_sector(ctx, L, 2.0, 11, nup=nup)
    lo, hi = g.extremal_bounds(sec)
    sigma = lo + 0.31 * (hi - lo)
    rng = np.random.default_rng(nrhs)
    b = rng.standard_normal((sec.dim, nrhs))
    f = g.factor(sec, sigma, precision=prec)
    x = f.solve(b, refine=True)
    r = b - sec.spmv(x, shift=sigma)
    a = max(abs(lo), abs(hi)) + abs(sigma)
    lim = 2e-14 * (a * np.linalg.norm(x, axis=0) + np.linalg.norm(b, axis=0))
    assert (np.linalg.norm(r, axis=0) <= lim).all()


def _refined_residual_is_small(ctx, L, nup, nrhs, scale=None, **kw):
    """The bound of test_refined_solve_leaves_a_small_residual, per column (each column's own scale)."""
    sec = g.build_sector(ctx, L, 2.0, 11, nup=nup)
    lo, hi = g.extremal_bounds(sec)
    sigma = lo + 0.31 * (hi - lo)
    b = np.random.default_rng(nrhs).standard_normal((sec.dim, nrhs))
    if scale is not None:
        b *= scale(sec.dim)[:, None]
    x = g.factor(sec, sigma, **kw).solve(b, refine=True)
    r = b - sec.spmv(x, shift=sigma)
    a = max(abs(lo), abs(hi)) + abs(sigma)
    lim = 2e-14 * (a * np.linalg.norm(x, axis=0) + np.linalg.norm(b, axis=0))
    assert (np.linalg.norm(r, axis=0) <= lim).all()


@pytest.mark.gpu
@pytest.mark.parametrize("L,nup,nrhs", [(14, 7, 1), (15, 7, 3), (15, 8, 16), (15, 7, 20), (16, 8, 31), (17, 8, 32)])
def test_fronts_of_several_solve_panels(ctx, L, nup, nrhs):
    """Panel steps and updates with and without padded right-hand sides, partial row blocks and last panels;
    Arnoldi steps of up to four and eight elements a thread, and longer ones (n nrhs / 152 / 512)."""
    _refined_residual_is_small(ctx, L, nup, nrhs)


@pytest.mark.gpu
@pytest.mark.parametrize("tc", [0, 1, 2])
@pytest.mark.parametrize("L,nup", [(10, 4), (13, 6), (15, 7)])
def test_trailing_updates_of_every_kind(ctx, L, nup, tc):
    """CUDA-core, 3xTF32 and 3xBF16 updates on trailing blocks that end inside a 128 x 64 tile."""
    _refined_residual_is_small(ctx, L, nup, 5, precision=g.MBL_PREC_FP32, tensor_cores=tc)


@pytest.mark.gpu
@pytest.mark.parametrize("L,nup,nrhs", [(9, 4, 1), (12, 6, 9), (14, 7, 17), (15, 7, 32)])
@pytest.mark.parametrize("span", [0, 40, 600])
def test_fp64_fronts_and_right_hand_sides_of_wide_range(ctx, L, nup, nrhs, span):
    """FP64 fronts and solves on fixed-point digits: right-hand sides whose entries span 2^span go through
    several passes of the digits, each on its own scale."""
    def scale(n):
        return np.exp2(-np.random.default_rng(span).uniform(0, span, n))
    _refined_residual_is_small(ctx, L, nup, nrhs, scale, precision=g.MBL_PREC_FP64)


@pytest.mark.gpu
@pytest.mark.parametrize("L,nup", [(11, 5), (12, 5), (12, 6), (13, 6)])
def test_extremal_bounds_against_a_dense_spectrum(ctx, L, nup):
    """The bounds stop at a residual of 1e-13 |H|, which bounds the eigenvalue's error; the dense solver adds
    some ulps times sqrt(n), below 1e-14 |H|: 2e-13 |H| in all.  Row counts that are no multiple of a warp's
    eight rows or of the four sets a lane group takes."""
    sec = g.build_sector(ctx, L, 1.5, 4, nup=nup)
    w = np.linalg.eigvalsh(sec.spmv(np.eye(sec.dim)))
    lo, hi = g.extremal_bounds(sec)
    assert max(abs(lo - w[0]), abs(hi - w[-1])) <= 2e-13 * max(abs(w[0]), abs(w[-1]))

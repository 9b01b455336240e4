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

"""The residual norm that a mixed V-cycle solve reports is that of the FP64 residual of the iterate it
returns, not of a residual rounded to FP32.

The outer residual carries FP64 values as FP32 pairs: products and sums to about 44 bits, so an entry is
off by some 1e-13 of sum |a_ij| |x_j|.  After one or two cycles that sum is at most a few hundred times
the residual's entries, and the norm is off by less than 1e-10 of itself; single rounding of the entries
(6e-8 each) shows at 1e-9 and above on meshes of some hundred rows.  The squares are summed by way of the
residual's bits, or in FP64 where these are very large or small: so also for right-hand sides scaled by 1e20
and 1e-24 (pairs carry these as accurately), a column of zeros, and more rows than one round of blocks."""
import numpy as np
import pytest
import scipy.sparse as sp

import meshgen
import paper_1505_03615_gb300 as L

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"
T = 1e-2



def _check(h, depth, nrhs, scale=1.0, zero=None):
    L.lbmg_assemble(h, T)
    rp, ci, M, S = L.lbmg_get_matrix(h, depth)
    n = rp.size - 1
    A = sp.csr_matrix((M + T * S, ci, rp), shape=(n, n))
    b = scale * (A @ np.random.default_rng(5).normal(size=(n, nrhs)))
    if zero is not None:
        b[:, zero] = 0.0
    nb = np.linalg.norm(b, axis=0)
    for cycles in (1, 2):
        x = torch.zeros((n, nrhs), dtype=torch.float64, device=DEV)
        code, st = L.lbmg_solve(h, torch.tensor(b, device=DEV), x, 1e-30, cycles, L.LBMG_MIXED)
        assert code == L.LBMG_NOT_CONVERGED and st.cycles == cycles
        true = np.linalg.norm(b - A @ x.cpu().numpy(), axis=0) / np.where(nb > 0, nb, 1.0)
        kept = np.array(st.rel_residual[:nrhs])
        assert np.all(np.abs(kept - true) <= 1e-10 * true), (kept, true)
    return n


@pytest.mark.parametrize("host", [0, 1])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4])
@pytest.mark.parametrize("sub,depth", [(1, 3), (2, 4)])
def test_reported_norm_is_that_of_the_fp64_residual(sub, depth, nrhs, host):
    V, F = meshgen.icosphere(sub, 1.0, 1e-3, 1)
    h = L.lbmg_build_hierarchy(V, F, depth, host_check=host, coarse_max=60)
    try:
        _check(h, depth, nrhs)
    finally:
        L.lbmg_destroy(h)


@pytest.mark.parametrize("scale,zero", [(1e20, None), (1e-24, None), (1.0, 1)])
def test_reported_norm_of_large_small_and_zero_residuals(scale, zero):
    V, F = meshgen.icosphere(2, 1.0, 1e-3, 1)
    h = L.lbmg_build_hierarchy(V, F, 4, coarse_max=60)
    try:
        for nrhs in (2, 3):
            _check(h, 4, nrhs, scale, zero)
    finally:
        L.lbmg_destroy(h)


def test_reported_norm_on_more_rows_than_one_round():
    V, F = meshgen.torus_knot_tube(2, 3, 1.0, 0.04, 1400, 100, 1e-6, 2)
    h = L.lbmg_build_hierarchy(V, F, 9)
    try:
        for nrhs in (1, 2, 4):
            assert _check(h, 9, nrhs) > 155_648
    finally:
        L.lbmg_destroy(h)

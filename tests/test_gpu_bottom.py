"""Mixed cycles and conjugate gradients whose one-block bottom (from global memory) reaches up to the
finest level.  The block sweeps that level from a zero start, so the caller has to zero it: whatever an
earlier call left in the work vectors must not enter the next one.

Two handles of the same meshes: the tiled sweeps of the default shapes (no one-block bottom), and one
with the finest level's sweep set by hand, which sends all levels to the one block.  They differ by the
order of FP32 additions inside a row, as the launch shapes do (1e-4 in the evaluated function after a few
sweeps or cycles); the second has solved for a right-hand side 1e6 times as large just before."""
import numpy as np
import pytest

import meshgen
import paper_1505_03615_gb300 as L

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"


def _pair(build):
    hs = [build(), build()]
    D = L.lbmg_levels(hs[0])[1]
    for h in hs:
        L.lbmg_assemble(h, 1e-2)
    L.lbmg_set_launch_shape(hs[1], D, L.LBMG_MIXED, 0, 4, 256)
    return hs, D


def _rhs(h, V, nrhs, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    f = torch.randn((V.shape[0], nrhs), dtype=torch.float64, device=DEV, generator=g)
    b = torch.zeros((L.lbmg_level_info(h, L.lbmg_levels(h)[1])[0], nrhs), dtype=torch.float64, device=DEV)
    L.lbmg_project_rhs(h, f, b)
    return b


def _close(hs, V, xs):
    """The functions, not their coefficients: those of nearly dependent functions are undetermined."""
    us = []
    for h, x in zip(hs, xs):
        u = torch.zeros((V.shape[0], x.shape[1]), dtype=torch.float64, device=DEV)
        L.lbmg_eval_vertices(h, x, u)
        us.append(u)
    assert torch.isfinite(us[1]).all()
    assert float((us[1] - us[0]).abs().max()) <= 1e-4 * float(us[0].abs().max())


@pytest.mark.parametrize("host", [0, 1])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4])
def test_conjugate_gradients_on_a_batch_start_from_zero(nrhs, host):
    meshes = [(*meshgen.icosphere(1, 1.0, 1e-3, 1), 3), (*meshgen.icosphere(2, 0.7, 1e-3, 2), 3)]
    V = np.concatenate([m[0] for m in meshes])
    hs, D = _pair(lambda: L.lbmg_build_batch(meshes))
    try:
        assert L.lbmg_level_info(hs[0], D)[0] <= L.lbmg_default_options().narrow_max
        b = _rhs(hs[0], V, nrhs, 1)
        for h in hs:
            L.lbmg_set_host_check(h, host)
        L.lbmg_solve_pcg(hs[1], 1e6 * _rhs(hs[0], V, nrhs, 2), torch.zeros_like(b), 1e-30, 2, L.LBMG_MIXED)
        for steps in (1, 2):
            xs = []
            for h in hs:
                x = torch.zeros_like(b)
                code, st = L.lbmg_solve_pcg(h, b, x, 1e-30, steps, L.LBMG_MIXED)
                assert code == L.LBMG_NOT_CONVERGED and st.cycles == steps
                xs.append(x)
            _close(hs, V, xs)
    finally:
        for h in hs:
            L.lbmg_destroy(h)


@pytest.mark.parametrize("opts", [dict(), dict(use_graphs=0), dict(nu1=2, nu2=0)])
def test_cycles_of_a_mesh_whose_bottom_does_not_fit_shared_memory_start_from_zero(opts):
    """The coarsest level (about 2000 rows) is beyond a block's shared memory, so the bottom, here the whole
    hierarchy, runs from global memory."""
    V, F = meshgen.icosphere(3, 1.0, 1e-3, 1)
    hs, D = _pair(lambda: L.lbmg_build_hierarchy(V, F, 5, coarse_max=2048, min_depth=4, narrow_max=10000, **opts))
    try:
        assert L.lbmg_levels(hs[0]) == (4, 5) and L.lbmg_level_info(hs[0], D)[0] <= 10000
        if opts.get("nu2", 2):   # the finest level's sweeps, transfers and the coarse solve in one launch
            assert L.lbmg_launch_counts(hs[1], L.LBMG_MIXED)[2] < L.lbmg_launch_counts(hs[0], L.LBMG_MIXED)[2]
        b = _rhs(hs[0], V, 3, 1)
        big = 1e6 * _rhs(hs[0], V, 3, 2)
        for solve in ("cycles", "cg"):
            xs = []
            for h in hs:
                x = torch.zeros_like(b)
                if solve == "cycles":
                    L.lbmg_vcycles(h, big, torch.zeros_like(b), 2, L.LBMG_MIXED)
                    L.lbmg_vcycles(h, b, x, 2, L.LBMG_MIXED)
                else:
                    L.lbmg_solve_pcg(h, big, torch.zeros_like(b), 1e-30, 2, L.LBMG_MIXED)
                    L.lbmg_solve_pcg(h, b, x, 1e-30, 2, L.LBMG_MIXED)
                xs.append(x)
            _close(hs, V, xs)
    finally:
        for h in hs:
            L.lbmg_destroy(h)

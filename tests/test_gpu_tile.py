"""The tiled Gauss-Seidel sweep (the default on levels of up to some ten thousand rows) against the
colour launches, which a launch shape set by hand selects.

Both update every row from the same values; only the order of the additions inside a row may differ.  So
they agree as the launch shapes do among one another (test_gpu_tune.py): 1e-11 relative in FP64 and 1e-4
in FP32 after a few sweeps, and whole cycles from zero to 1e-9 and 1e-4 in the evaluated function."""
import numpy as np
import pytest

import meshgen
import paper_1505_03615_gb300 as L

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"

MESHES = {
    "knot": lambda: (*meshgen.torus_knot_tube(2, 3, 1.0, 0.12, 48, 8, 1e-6, 3), 5),
    "sheet": lambda: (*meshgen.double_sheet(60, 0.05, 6), 6),           # rows of more than 32 entries
    "twoparts": lambda: (*meshgen.torus_knot_tube(2, 3, 1.0, 0.04, 600, 60, 1e-6, 2), 8),   # > 40,000 rows
}


def _pair(name, **opts):
    """Two handles of one mesh: the tiled sweep where it is the default, and the colour launches."""
    if name == "batch":
        meshes = meshgen.batch_mix(3, 2_000, 12_000, 5)
        hs = [L.lbmg_build_batch(meshes, **opts) for _ in range(2)]
    else:
        V, F, depth = MESHES[name]()
        hs = [L.lbmg_build_hierarchy(V, F, depth, **opts) for _ in range(2)]
    d0, D = L.lbmg_levels(hs[0])
    for h in hs:
        L.lbmg_assemble(h, 1e-3)
    for d in range(d0 + 1, D + 1):
        for prec in (L.LBMG_FP64, L.LBMG_MIXED):
            L.lbmg_set_launch_shape(hs[1], d, prec, 0, 4, 256)
    return hs, d0, D


def _rel(a, b):
    return float((a - b).abs().max() / b.abs().max())


@pytest.mark.parametrize("name", ["knot", "sheet", "twoparts", "batch"])
def test_tiled_sweeps_match_the_colour_launches(name):
    hs, d0, D = _pair(name)
    g = torch.Generator(device=DEV)
    g.manual_seed(1)
    try:
        for d in range(d0 + 1, D + 1):
            n = L.lbmg_level_info(hs[0], d)[0]
            for nrhs in (1, 2, 3, 4):
                xr = torch.randn((n, nrhs), dtype=torch.float64, device=DEV, generator=g)
                x0 = torch.rand((n, nrhs), dtype=torch.float64, device=DEV, generator=g)
                b = torch.zeros_like(xr)
                L.lbmg_residual(hs[0], d, b, xr, b)
                b = -b   # a right-hand side in the range of A
                for prec, tol in ((L.LBMG_FP64, 1e-11), (L.LBMG_MIXED, 1e-4)):
                    for sweeps in (1, 2):
                        xs = []
                        for h in hs:
                            x = x0.clone()
                            L.lbmg_smooth(h, d, b, x, sweeps, prec)
                            xs.append(x)
                        assert _rel(xs[0], xs[1]) <= tol, (d, nrhs, prec, sweeps)
    finally:
        for h in hs:
            L.lbmg_destroy(h)


@pytest.mark.parametrize("nu", [(2, 2), (1, 2), (2, 1), (3, 3), (0, 2), (2, 0)])
@pytest.mark.parametrize("graphs", [1, 0])
def test_cycles_with_tiled_sweeps_match(nu, graphs):
    """Odd and missing sweeps too: the vector changes buffers with every tiled sweep."""
    hs, d0, D = _pair("knot", nu1=nu[0], nu2=nu[1], use_graphs=graphs, min_depth=1)
    try:
        n = L.lbmg_level_info(hs[0], D)[0]
        V = MESHES["knot"]()[0]
        rhs = torch.zeros((n, 3), dtype=torch.float64, device=DEV)
        L.lbmg_project_rhs(hs[0], torch.tensor(V, device=DEV), rhs)
        for prec, tol in ((L.LBMG_FP64, 1e-9), (L.LBMG_MIXED, 1e-4)):
            us = []
            for h in hs:
                x, u = torch.zeros_like(rhs), torch.zeros((V.shape[0], 3), dtype=torch.float64, device=DEV)
                L.lbmg_vcycles(h, rhs, x, 3, prec)
                L.lbmg_eval_vertices(h, x, u)
                us.append(u)
            assert _rel(us[0], us[1]) <= tol
    finally:
        for h in hs:
            L.lbmg_destroy(h)


def test_a_nan_stays_where_the_colour_launches_leave_it():
    hs, d0, D = _pair("knot")
    try:
        n = L.lbmg_level_info(hs[0], D)[0]
        b = torch.ones((n, 3), dtype=torch.float64, device=DEV)
        b[n // 3, 1] = float("nan")
        b[n // 2, 2] = float("inf")
        out = []
        for h in hs:
            x = torch.zeros_like(b)
            L.lbmg_smooth(h, D, b, x, 1, L.LBMG_FP64)
            out.append(torch.isfinite(x))
        assert torch.equal(out[0], out[1]) and not out[0].all()
    finally:
        for h in hs:
            L.lbmg_destroy(h)

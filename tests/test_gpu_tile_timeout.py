"""Bounded waits of the tiled sweep that run out.  The step barrier is told to wait for one arrival that
never comes: every warp gives up as a whole after 10 ms, the kernel sets the status word and returns, the
host reports LBMG_DEVICE_TIMEOUT once, and the handle and the device keep working (with colour launches,
since the missing arrival belongs to the handle)."""
import pytest

import meshgen
import paper_1505_03615_gb300 as L

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"
DEPTH = 6


def _handles(**opts):
    V, F = meshgen.torus(1.0, 0.3, 80, 30)
    hs = [L.lbmg_build_hierarchy(V, F, DEPTH, barrier_phantoms=p, **opts) for p in (1, 0)]
    for h in hs:
        L.lbmg_assemble(h, 1e-2)
    rhs = torch.zeros((L.lbmg_level_info(hs[0], DEPTH)[0], 3), dtype=torch.float64, device=DEV)
    L.lbmg_project_rhs(hs[0], torch.tensor(V, dtype=torch.float64, device=DEV), rhs)
    return hs, rhs


def _colour_launches(h):
    d0, D = L.lbmg_levels(h)
    for d in range(d0 + 1, D + 1):
        for prec in (L.LBMG_FP64, L.LBMG_MIXED):
            L.lbmg_set_launch_shape(h, d, prec, 0, 4, 256)


@pytest.mark.parametrize("host", [0, 1])
@pytest.mark.parametrize("prec", [L.LBMG_FP64, L.LBMG_MIXED])
@pytest.mark.parametrize("solve", [L.lbmg_solve, L.lbmg_solve_pcg])
def test_a_solve_whose_steps_wait_in_vain_reports_it(solve, prec, host):
    hs, rhs = _handles(host_check=host)
    try:
        assert solve(hs[0], rhs, torch.zeros_like(rhs), 1e-6, 1000, prec)[0] == L.LBMG_DEVICE_TIMEOUT
        _colour_launches(hs[0])
        for h in hs:
            code, st = solve(h, rhs, torch.zeros_like(rhs), 1e-6, 1000, prec)
            assert code == L.LBMG_OK and st.converged
    finally:
        for h in hs:
            L.lbmg_destroy(h)

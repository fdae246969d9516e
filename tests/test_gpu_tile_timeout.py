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


def _expires(call):
    with pytest.raises(L.LbmgError) as e:
        call()
    assert e.value.code == L.LBMG_DEVICE_TIMEOUT


@pytest.mark.parametrize("prec", [L.LBMG_FP64, L.LBMG_MIXED])
def test_calls_that_wait_report_it_and_clear_it(prec):
    hs, rhs = _handles(use_graphs=0, host_check=1)
    h = hs[0]
    try:
        b, x = rhs.cpu().numpy(), rhs.cpu().numpy() * 0
        calls = [lambda: L.lbmg_smooth(h, DEPTH, b, x, 1, prec), lambda: L.lbmg_vcycles(h, b, x, 1, prec),
                 lambda: L.lbmg_autotune(h, 3, prec, 1)]
        for call in calls:
            _expires(call)
        _colour_launches(h)
        for call in calls[:2]:
            assert call() == L.LBMG_OK
    finally:
        for q in hs:
            L.lbmg_destroy(q)


@pytest.mark.parametrize("opts", [dict(), dict(host_check=1), dict(persistent=1)])
def test_the_next_solve_reports_it_once_for_a_call_that_does_not_wait(opts):
    hs, rhs = _handles(**opts)
    h = hs[0]
    try:
        L.lbmg_smooth(h, DEPTH, rhs, torch.zeros_like(rhs), 1, L.LBMG_FP64)
        if not opts.get("persistent"):   # (its own barrier has the missing arrival too)
            _colour_launches(h)
        assert L.lbmg_solve(h, rhs, torch.zeros_like(rhs), 1e-6, 1000, L.LBMG_FP64)[0] == L.LBMG_DEVICE_TIMEOUT
        if not opts.get("persistent"):
            assert L.lbmg_solve(h, rhs, torch.zeros_like(rhs), 1e-6, 1000, L.LBMG_FP64)[0] == L.LBMG_OK
    finally:
        for q in hs:
            L.lbmg_destroy(q)


@pytest.mark.parametrize("host", [0, 1])
def test_conjugate_gradients_on_a_batch_report_it(host):
    meshes = [(*meshgen.torus(1.0, 0.3, 40, 16), 5), (*meshgen.icosphere(3, 1.0, 1e-3, 1), 5)]
    hs = [L.lbmg_build_batch(meshes, barrier_phantoms=p, host_check=host) for p in (1, 0)]
    try:
        for h in hs:
            L.lbmg_assemble(h, 1e-2)
        b = torch.ones((L.lbmg_level_info(hs[0], L.lbmg_levels(hs[0])[1])[0], 2), dtype=torch.float64, device=DEV)
        codes = [L.lbmg_solve_pcg(h, b, torch.zeros_like(b), 1e-30, 2, L.LBMG_FP64)[0] for h in hs]
        assert codes == [L.LBMG_DEVICE_TIMEOUT, L.LBMG_NOT_CONVERGED]
        _colour_launches(hs[0])
        assert L.lbmg_solve_pcg(hs[0], b, torch.zeros_like(b), 1e-30, 2, L.LBMG_FP64)[0] == L.LBMG_NOT_CONVERGED
    finally:
        for h in hs:
            L.lbmg_destroy(h)


def test_eigenpairs_and_training_report_it():
    hs, rhs = _handles()
    h = hs[0]
    try:
        X0 = torch.rand((rhs.shape[0], 2), dtype=torch.float64, device=DEV)
        order = [[0], [1]]
        _expires(lambda: L.lbmg_eigs(h, X0.clone(), 1e-6, 3))
        _expires(lambda: L.lbmg_learned_collect(h, rhs, 0, 2))
        _expires(lambda: L.lbmg_learned_loss_grad(h, rhs))
        _colour_launches(h)
        assert L.lbmg_eigs(h, X0.clone(), 1e-30, 2)[0] == L.LBMG_NOT_CONVERGED
        with pytest.raises(L.LbmgError) as e:   # the expired call has stored no samples
            L.lbmg_learned_train(h, order, 1e-3)
        assert e.value.code == 1
        L.lbmg_learned_collect(h, rhs, 0, 2)
        assert len(L.lbmg_learned_train(h, order, 1e-3)) == 2
    finally:
        for q in hs:
            L.lbmg_destroy(q)

"""Conjugate gradients for one to four right-hand sides, on one mesh and on a batch whose meshes have from
a few rows of a colour to several work items of them, with the loop in the graph and with the host reading the
norms.  Step by step, mesh by mesh and column by column:
- the residual norm that the iteration keeps is that of b - A x, formed from the matrices on the host.  The two
  differ by what a few additions and products of vectors no larger than the largest residual so far round off:
  1e-9 of that residual in FP64, 1e-6 with the products in FP32 pairs (46 bits; the kept norm is relative to b);
- the error in the A-norm never grows (each step minimises it along p), to 1e-9 and 1e-4 of itself;
- a column that is zero stays zero."""
import numpy as np
import pytest
import scipy.sparse as sp

import meshgen
import paper_1505_03615_gb300 as L

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"
T = 1e-2


def _build(name):
    if name == "batch":
        return L.lbmg_build_batch([(*meshgen.icosphere(1, 1.0, 1e-3, 1), 3), *meshgen.batch_mix(3, 2_000, 12_000, 5),
                                   (*meshgen.double_sheet(8, 0.05, 5, 0.5, 1e-6, 4), 5)])
    return L.lbmg_build_hierarchy(*meshgen.icosphere(*((1,) if name == "tiny" else (5,)), 1.0, 1e-3, 1),
                                  3 if name == "tiny" else 6)


@pytest.mark.parametrize("name", ["tiny", "sphere", "batch"])
@pytest.mark.parametrize("precision,kept_tol,err_tol", [(L.LBMG_FP64, 1e-9, 1e-9), (L.LBMG_MIXED, 1e-6, 1e-4)])
def test_steps_keep_the_true_residual_and_shrink_the_error(name, precision, kept_tol, err_tol):
    h = _build(name)
    try:
        L.lbmg_assemble(h, T)
        D = L.lbmg_levels(h)[1]
        rp, ci, M, S = L.lbmg_get_matrix(h, D)
        n = rp.size - 1
        A = sp.csr_matrix((M + T * S, ci, rp), shape=(n, n))
        inst = L.lbmg_row_instances(h, D) if name == "batch" else np.zeros(n, dtype=int)
        user = np.argsort(inst, kind="stable")   # vectors hold mesh after mesh
        A, inst = A[user][:, user], inst[user]
        meshes = range(inst.max() + 1)
        xt = np.random.default_rng(1).normal(size=(n, 4))
        for nrhs in (1, 2, 3, 4):
            xe = xt[:, :nrhs].copy()
            if nrhs > 2:
                xe[:, 1] = 0.0
            b = A @ xe
            for host in (0, 1):
                L.lbmg_set_host_check(h, host)
                peak = np.ones((len(meshes), nrhs))
                err = np.array([np.einsum("ij,ij->j", xe[inst == i], b[inst == i]) for i in meshes])
                for steps in (1, 2, 3, 4):
                    x = torch.zeros((n, nrhs), dtype=torch.float64, device=DEV)
                    code, st = L.lbmg_solve_pcg(h, torch.tensor(b, device=DEV), x, 1e-30, steps, precision)
                    assert code == L.LBMG_NOT_CONVERGED and st.cycles == steps
                    kept = L.lbmg_instance_residuals(h, nrhs) if name == "batch" else np.array([st.rel_residual[:nrhs]])
                    xh = x.cpu().numpy()
                    r = b - A @ xh
                    e = xe - xh
                    Ae = A @ e
                    peak = np.maximum(peak, kept)
                    for i in meshes:
                        rows = inst == i
                        nb = np.linalg.norm(b[rows], axis=0)
                        true = np.linalg.norm(r[rows], axis=0) / np.where(nb > 0, nb, 1.0)
                        assert np.all(np.abs(kept[i] - true) <= kept_tol * peak[i])
                        now = np.einsum("ij,ij->j", e[rows], Ae[rows])
                        assert np.all(now <= err[i] * (1 + err_tol))
                        err[i] = now
                    assert nrhs < 3 or not xh[:, 1].any()
    finally:
        L.lbmg_destroy(h)

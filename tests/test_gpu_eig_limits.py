"""Eigensolves cut off after one, two or three iterations, on two and three levels: a
coarse level tests its pairs before it updates them, so after one iteration its
selection comes from the Ritz values alone.  The hierarchy is kept and reported
unconverged, the counts stay within 1..nev, and any coarse space of that kind is a
valid preconditioner: PCG reaches its tolerance (true residual within twice 1e-8).
"""
import numpy as np
import pytest

import synthetic_inputs as si
from oracle import fem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402

NEV = 6


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("levels", [2, 3])
@pytest.mark.parametrize("maxit", [1, 2, 3])
def test_iteration_limits(maxit, levels, precision):
    # memory that held other numbers before: nothing may be left to what a buffer happens to hold
    junk = [torch.full((1 << k,), 0x7f0f7f0f, dtype=torch.int32, device="cuda") for k in range(7, 24)]
    del junk
    torch.cuda.empty_cache()
    k = si.channels_2d(48, 12, 1e4, seed=1)
    G = pkg.Hierarchy((48, 48), torch.tensor(k, device="cuda"), (6, 6), 2, levels, (2, 2), NEV, 0.3,
                      precision=precision, eig_maxit=maxit, fp32_start_iters=1, eig_tol=1e-12,
                      allow_eig_unconverged=True)
    st = G.stats()
    fine = levels - 1
    assert G.setup_status == -4
    assert st["eig_iters_max"][fine] == maxit and st["eig_iters_total"][fine] <= 36 * maxit
    assert 1 <= st["eig_unconverged"][fine] <= 36
    assert 0 <= st["m_min"][fine] and 1 <= st["m_max"][fine] <= NEV
    if levels == 3:
        assert st["eig_iters_max"][1] <= maxit and st["eig_unconverged"][1] <= 9
        assert 0 <= st["m_min"][1] and 1 <= st["m_max"][1] <= NEV
        for i in range(9):
            theta, m = G.eigenvalues(1, i)
            assert m == min(NEV, int((theta < 0.3).sum())) if maxit == 1 else 0 <= m <= NEV
    mesh = fem.Mesh((48, 48), 0b1)
    A, b = fem.assemble_system(mesh, k), fem.load_vector(mesh)
    x, _, rel = G.solve(torch.tensor(b, device="cuda"), tol=1e-8, maxit=3000)
    assert rel < 1e-8 and np.linalg.norm(b - A @ x.cpu().numpy()) <= 2e-8 * np.linalg.norm(b)
    G.close()

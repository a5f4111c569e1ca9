"""Eigensolves of coarse subdomains whose generating systems are nearly dependent: two
blocks of columns of strips, block functions of degree 3, wide overlap; hundreds of null
pivots and others just above the bound that drops them.  The solves apply a dense
pseudo-inverse there, and every column of it has to be the backward stable solution for
its unit vector: an inverse whose entries come from different solves multiplies the
errors by the condition number.

The rounding floor of such a pencil lies a little below the accepted residual (the root
of the tolerance, 1e-3), so a few of the 18 subdomains may stay above it: at most two.
Every other one has to reach it, for the selected pairs.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("precision,start", [(0, None), (1, 12)])
@pytest.mark.parametrize("seed", [3096340, 0, 1])
def test_solves_of_nearly_dependent_generators_reach_their_floor(seed, precision, start):
    rng = np.random.default_rng(seed)
    n = (84, 85)
    k = 10.0 ** rng.uniform(-0.5, 0.5, n[0] * n[1])
    T = np.zeros((k.size, 3))
    T[:, :2] = k[:, None]
    T[:, 2] = 0.3 * k * rng.uniform(-1, 1, k.size)
    G = pkg.Hierarchy(n, torch.tensor(T, device="cuda"), (12, 3), 3, 3, (2, 1), 23, 0.9, dirichlet_faces=0b0110,
                      precision=precision, block_p=32, blf=3, fp32_start_iters=start, allow_eig_unconverged=True)
    st = G.stats()
    assert st["null_pivots"][1] > 300
    assert st["eig_unconverged"][0] == st["eig_unconverged"][2] == 0 and st["eig_unconverged"][1] <= 2, st
    missed = 0
    for j in range(st["subdomains"][1]):
        m = G.eigenvalues(1, j)[1]
        missed += bool(np.asarray(G.eigen_residuals(1, j)[0][:m]).max(initial=0.0) > 1e-3)
    assert missed <= 2
    G.close()

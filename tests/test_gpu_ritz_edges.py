"""Rayleigh-Ritz at the block sizes where its kernel changes form: 5 to 32
columns, odd sizes (padded by one), and each side of the register block sizes
12, 16 and 20 of the Cholesky factor.  Channels of one contrast give groups of
nearly equal eigenvalues (0.1605, 0.1611, 0.1616; 0.99658 three times), a
rough coefficient gives separated ones.

Reference: the oracle's dense eigenvalues.  Eigenvalue errors are second order
in the residual tolerance 1e-7, so the library's stated bound applies, 1e-6
relative with an absolute floor for eigenvalues near zero.
"""
import numpy as np
import pytest

import synthetic_inputs as si
from oracle import fem, method

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402

ETA = 0.9
_ORACLE = {}


def _eigenvalues(field):
    if field not in _ORACLE:
        if field == "rough":
            kap = 10.0 ** np.random.default_rng(7).uniform(-1, 1, 24 * 24)
        else:
            kap = si.channels_2d(24, 6, 1e4, seed=2)
        H = method.Hierarchy(fem.Mesh((24, 24), 0b1), kap, (2, 2), 2, 2, (1, 1), 30, ETA)
        _ORACLE[field] = kap, H.eigenvalues(1)
    return _ORACLE[field]


@pytest.mark.parametrize("nev", [1, 8, 9, 12, 13, 16, 17, 23, 24])
@pytest.mark.parametrize("field", ["rough", "channels"])
def test_eigenvalues_at_block_edges(field, nev):
    kap, lam = _eigenvalues(field)
    G = pkg.Hierarchy((24, 24), torch.tensor(kap, device="cuda"), (2, 2), 2, 2, (1, 1), nev, ETA, precision=0,
                      block_p=32 if nev == 24 else 0, eig_tol=1e-7)
    for i, ref in enumerate(lam):
        theta, m = G.eigenvalues(1, i)
        n = min(m, len(theta), len(ref))
        assert n >= 1
        t, r = np.asarray(theta[:n]), np.asarray(ref[:n])
        assert (np.abs(t - r) <= 1e-6 * np.maximum(r, 1e-3 * ETA)).all(), (i, t, r)
    G.close()

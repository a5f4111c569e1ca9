"""Eigensolves whose block spans the whole range of the pencil's right-hand side:
subdomains of a few dozen nodes, where the block holds every direction and its last
Ritz values of the inverse are rounding errors; and coarse levels of as many own
generators as the block has columns.

Reference: the oracle's dense eigenvalues and selection on the fine level, counts
exactly, eigenvalues to 1e-6 relative with a floor of 1e-3 eta (the library's stated
bound at eigen-residuals of 1e-6 and below), with eigenvalues that keep 1e-4 eta
away from eta; no pair may be lost (1e300) below the selected ones;
PCG to 1e-8 with a true residual within twice that.  The set-up is run several times:
nothing may depend on what memory held.
"""
import functools

import numpy as np
import pytest

from oracle import fem, method

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402

# mesh, subdomains, overlap, nev, eta, coarse groups, decades of the coefficient on each side of 1
CASES = {"strips": ((44, 13), (12, 12), 2, 24, 0.3, (3, 2), 1.0), "squares": ((20, 20), (5, 5), 1, 16, 0.3, (2, 2), 1.0),
         "cubes": ((8, 8, 8), (4, 4, 4), 1, 16, 0.3, (2, 2, 2), 1.0), "six": ((9, 7), (3, 2), 1, 24, 0.9, (1, 1), 1.0),
         "thin": ((26, 4), (8, 2), 1, 5, 0.9, (2, 1), 2.0)}


@functools.lru_cache(maxsize=None)
def _reference(name):
    n, parts, overlap, nev, eta, group, decades = CASES[name]
    k = 10.0 ** np.random.default_rng(len(name)).uniform(-decades, decades, int(np.prod(n)))
    H = method.Hierarchy(fem.Mesh(n, 0b1), k, parts, overlap, 2, (1,) * len(n), nev, eta)
    lam = H.eigenvalues(1)
    assert min(float(np.abs(np.asarray(v) - eta).min()) for v in lam) > 1e-4 * eta
    return k, lam, H.counts(1)


@pytest.mark.parametrize("precision,start", [(0, 0), (1, 0), (1, 6), (1, 20)])
@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("block", ["least", "default", "widest"])
def test_blocks_as_wide_as_the_subdomain(name, precision, start, block):
    n, parts, overlap, nev, eta, _, _ = CASES[name]
    k, lam, counts = _reference(name)
    kd = torch.tensor(k, device="cuda")
    for _ in range(3):
        G = pkg.Hierarchy(n, kd, parts, overlap, 2, (1,) * len(n), nev, eta, precision=precision, fp32_start_iters=start,
                          block_p={"least": nev + 1, "default": 0, "widest": 32}[block])
        for i, ref in enumerate(lam):
            theta, m = G.eigenvalues(1, i)
            assert m == counts[i], (i, m, counts[i], theta[:4])
            t, r = np.asarray(theta[:m]), np.asarray(ref[:m])
            assert (np.abs(t - r) <= 1e-6 * np.maximum(r, 1e-3 * eta)).all(), (i, t, r)
        G.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", ["cubes", "squares", "strips"])
def test_three_levels_of_small_subdomains(name, precision):
    n, parts, overlap, nev, eta, group, _ = CASES[name]
    k, _, counts = _reference(name)
    mesh = fem.Mesh(n, 0b1)
    A, b = fem.assemble_system(mesh, k), fem.load_vector(mesh)
    dims = set()
    for _ in range(3):
        G = pkg.Hierarchy(n, torch.tensor(k, device="cuda"), parts, overlap, 3, group, nev, eta, precision=precision,
                          allow_eig_unconverged=True)
        st = G.stats()
        assert st["level_dim"][1] == sum(counts)
        dims.add(st["level_dim"][0])
        x, _, rel = G.solve(torch.tensor(b, device="cuda"), tol=1e-8, maxit=500)
        assert rel < 1e-8 and np.linalg.norm(b - A @ x.cpu().numpy()) <= 2e-8 * np.linalg.norm(b)
        G.close()
    assert len(dims) == 1, dims

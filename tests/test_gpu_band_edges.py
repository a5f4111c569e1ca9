"""Band solves at the sizes where the tiled kernels can go wrong: orders around
tile edges (1, 31, 32, 33, ...), half-bandwidths around multiples of the tile,
full bandwidth, problems of unequal order in one batch, one to 32 right-hand
sides.

Reference: numpy's dense FP64 solve of the same matrices.  The matrices are
diagonally dominant with off-diagonal row sums at most 1 against a diagonal of
at least 2, so their condition numbers are below 3 and the solves stay within a
few hundred rounding errors: relative error <= 1e-12 in FP64 (1e-16 x 1e3 rows
x a safety factor of 10) and <= 1e-4 in FP32 (the bound of the parity tests).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402

# (orders of the batch, half-bandwidth)
SHAPES = [([1], 0), ([2, 1], 1), ([31, 32, 33], 5), ([64, 65, 40], 31), ([97, 96, 70], 32), ([130, 129], 33),
          ([200, 161, 64], 45), ([150], 64), ([260, 180], 65), ([300, 299], 100), ([170, 33], 169), ([500], 381),
          ([321] * 5, 36)]


def _spd(n, bw, rng):
    A = np.zeros((n, n))
    for d in range(1, min(bw, n - 1) + 1):
        v = rng.uniform(-1.0, 1.0, n - d) / (2.0 * max(1, bw))
        A[np.arange(d, n), np.arange(n - d)] = v
        A[np.arange(n - d), np.arange(d, n)] = v
    return A + np.diag(2.0 + rng.uniform(0.0, 1.0, n))


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-4)])
@pytest.mark.parametrize("shape", range(len(SHAPES)))
def test_band_solve_at_tile_edges(shape, precision, tol):
    orders, bw = SHAPES[shape]
    rng = np.random.default_rng(100 + shape)
    nmax = max(orders)
    A = np.zeros((len(orders), nmax, nmax))
    for k, n in enumerate(orders):
        A[k, :n, :n] = _spd(n, bw, rng)
    bb = pkg.BandBatch(torch.tensor(A, device="cuda"), orders, bw, precision=precision)
    for nrhs in (1, 2, 3, 4, 5, 7, 8, 12, 16, 17, 20, 21, 32):
        B = rng.standard_normal((len(orders), nmax, nrhs))
        X = bb.solve(torch.tensor(B, device="cuda")).cpu().numpy()
        for k, n in enumerate(orders):
            ref = np.linalg.solve(A[k, :n, :n], B[k, :n])
            err = np.linalg.norm(X[k, :n] - ref) / np.linalg.norm(ref)
            assert err <= tol, (orders, bw, nrhs, k, err)
    bb.close()

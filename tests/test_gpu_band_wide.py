"""FP64 factorisations whose update of one tile column has more than 65535
tiles (362 or more tile rows below the diagonal: half-bandwidths above
11,552), beyond one grid dimension: a band and a dense matrix.

Reference: the solution is chosen and the right-hand side formed from it in
FP64.  The matrices are diagonally dominant, off-diagonal row sums at most 1
against a diagonal of at least 2, so their condition numbers are below 3; a
backward error of n rounding units gives at most 3 x 1.2e4 x 1.1e-16 = 4e-12,
and rounding errors of a sum grow like its square root: bound 1e-12, as for the
small matrices.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402


# 364 tile rows: 362 off-diagonal tiles a column (a band), 363 (all of them: dense)
@pytest.mark.parametrize("n,bw", [(32 * 364, 32 * 362), (32 * 364, 32 * 364)])
def test_fp64_factor_of_a_band_wider_than_one_grid_dimension(n, bw):
    gen = torch.Generator(device="cuda").manual_seed(5)
    f64 = dict(device="cuda", dtype=torch.float64)
    A = torch.rand((n, n), generator=gen, **f64).sub_(0.5)
    A.tril_(-1).triu_(-bw)
    A.add_(A.T.clone()).div_(n)
    A.diagonal().copy_(2.0 + torch.rand(n, generator=gen, **f64))
    bb = pkg.BandBatch(A[None], [n], bw, precision=0)
    for nrhs in (1, 5):
        x = torch.randn((n, nrhs), generator=gen, **f64)
        y = bb.solve((A @ x)[None].contiguous())[0]
        err = (torch.linalg.norm(y - x) / torch.linalg.norm(x)).item()
        assert err <= 1e-12, (nrhs, err)
    bb.close()

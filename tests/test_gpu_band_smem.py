"""Band solves whose dynamic shared memory ends just below 48 KB, where the
kernels' static arrays take a launch over the amount that needs no opt-in:
FP64 solves of several columns at 16, 32 and 64 tiles a row (4, 2 and 1 columns
a block), the FP64 one-column solve of a diagonal matrix of 51 tile rows, and the
one-column solves without a tile ring at 188 and 192 tile rows.

Reference: a chosen solution, the right-hand side formed from it in FP64; the
matrices and the bounds are those of the band solves at tile edges (diagonally
dominant, condition below 3: 1e-12 in FP64, 1e-4 in FP32).
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("count,n,bw,nrhs,precision", [
    (29, 520, 470, 32, 0), (15, 1030, 980, 32, 0), (1, 2060, 2000, 3, 0), (2, 1620, 0, 1, 0),
    (2, 6010, 400, 1, 0), (2, 6140, 400, 1, 1)])
def test_band_solve_near_the_default_shared_memory_limit(count, n, bw, nrhs, precision):
    gen = torch.Generator(device="cuda").manual_seed(n + bw)
    f64 = dict(device="cuda", dtype=torch.float64)
    A = torch.rand((count, n, n), generator=gen, **f64).sub_(0.5).tril_(-1).triu_(-bw).div_(max(1, bw))
    A.add_(A.transpose(1, 2).clone())
    A.diagonal(0, 1, 2).copy_(2.0 + torch.rand((count, n), generator=gen, **f64))
    x = torch.randn((count, n, nrhs), generator=gen, **f64)
    bb = pkg.BandBatch(A, [n] * count, bw, precision=precision)
    y = bb.solve((A @ x).contiguous())
    err = (torch.linalg.norm(y - x) / torch.linalg.norm(x)).item()
    assert err <= (1e-4 if precision else 1e-12), err
    bb.close()

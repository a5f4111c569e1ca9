"""One-column band solves on small and large batches: wide FP64 bands go through a
tile ring in shared memory while their blocks take at most two rounds over the
SMs and without a ring beyond, FP32 ones through the split of a step's tiles.

Reference: a chosen solution, the right-hand side formed from it in FP64;
diagonally dominant matrices (condition below 3), the bounds of the band solves at
tile edges: 1e-12 in FP64, 1e-4 in FP32.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-4)])
@pytest.mark.parametrize("count", [20, 304, 305, 640])
@pytest.mark.parametrize("orders,bw", [([140, 97, 128, 33], 90), ([200, 193, 64, 1], 157), ([330, 289, 320], 300)])
def test_one_column_solve(orders, bw, count, precision, tol):
    n = max(orders)
    sizes = [orders[k % len(orders)] for k in range(count)]
    gen = torch.Generator(device="cuda").manual_seed(bw + count)
    f64 = dict(device="cuda", dtype=torch.float64)
    A = torch.rand((count, n, n), generator=gen, **f64).sub_(0.5).tril_(-1).triu_(-bw).div_(bw)
    A.add_(A.transpose(1, 2).clone())
    A.diagonal(0, 1, 2).copy_(2.0 + torch.rand((count, n), generator=gen, **f64))
    inside = torch.arange(n, device="cuda")[None, :] < torch.tensor(sizes, device="cuda")[:, None]
    A.mul_((inside[:, :, None] & inside[:, None, :]).to(torch.float64))
    x = (torch.randn((count, n), generator=gen, **f64) * inside)[:, :, None]
    bb = pkg.BandBatch(A, sizes, bw, precision=precision)
    y = bb.solve((A @ x).contiguous()) * inside[:, :, None]
    err = ((y - x).flatten(1).norm(dim=1) / x.flatten(1).norm(dim=1)).max().item()
    assert err <= tol, err
    bb.close()

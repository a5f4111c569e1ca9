"""Band solves of several columns on batches that fill the chip, where the
number of problems decides the kernel and the columns a block takes.

With FP32 factors the dispatch chooses between a warp per few columns (ws: 16
columns a block up to two tiles of half-bandwidth, 20 beyond) and a split of the
tiles' columns over 4 or 8 warps (ks, 4 J columns a block): few problems take J
= 1, 160 or more take J = 1, 2, 3, 4, 5 for up to 4, 8, 12, 16, 20 columns and two
even groups beyond 20; an odd number of columns is not 16-byte aligned and
takes ks at every J.  With FP64 factors a block takes 4, 2 or 1 columns from 228
blocks on: the batches of 20, 70, 160 and more cover each.  The orders of a batch
differ (ends of tiles, one row, fewer rows than the band), so its problems have
different numbers of tile rows and bands.

Reference: a chosen solution, the right-hand side formed from it in FP64.  The
matrices are diagonally dominant, off-diagonal row sums at most 1 against a
diagonal of at least 2 (condition below 3): relative error <= 1e-12 in FP64
(1e-16 x 1e3 rows x a safety factor of 10) and <= 1e-4 in FP32, the bounds of
the band solves at tile edges.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402

# half-bandwidths of 1, 2, 3, 4, 6, 7 and 12 tiles; the orders of a batch in turn
BANDS = {20: (150, 33, 64, 97, 1, 129), 45: (150, 65, 33, 96, 161), 96: (193, 97, 40, 160, 128),
         110: (200, 129, 161, 64), 180: (260, 192, 225, 33), 223: (290, 257, 32, 224), 380: (450, 416, 385, 97)}
COLUMNS = (2, 4, 5, 7, 8, 10, 12, 13, 15, 16, 17, 18, 20, 21, 24, 28, 32)


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-4)])
@pytest.mark.parametrize("count", [20, 70, 160, 320, 620])
@pytest.mark.parametrize("bw", sorted(BANDS))
def test_band_solve_columns(bw, count, precision, tol):
    if count > 320 and bw > 110:
        pytest.skip("the same choices as 320 problems")
    orders = [BANDS[bw][k % len(BANDS[bw])] for k in range(count)]
    n = max(orders)
    gen = torch.Generator(device="cuda").manual_seed(1000 * bw + count)
    f64 = dict(device="cuda", dtype=torch.float64)
    A = torch.rand((count, n, n), generator=gen, **f64).sub_(0.5).tril_(-1).triu_(-bw).div_(bw)
    A.add_(A.transpose(1, 2).clone())
    A.diagonal(0, 1, 2).copy_(2.0 + torch.rand((count, n), generator=gen, **f64))
    inside = torch.arange(n, device="cuda")[None, :] < torch.tensor(orders, device="cuda")[:, None]
    A.mul_((inside[:, :, None] & inside[:, None, :]).to(torch.float64))
    bb = pkg.BandBatch(A, orders, bw, precision=precision)
    for nrhs in COLUMNS:
        x = torch.randn((count, n, nrhs), generator=gen, **f64) * inside[:, :, None]
        y = bb.solve((A @ x).contiguous()) * inside[:, :, None]
        err = ((y - x).flatten(1).norm(dim=1) / x.flatten(1).norm(dim=1)).max().item()
        assert err <= tol, (nrhs, err)
    bb.close()

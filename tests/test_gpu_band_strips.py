"""One-column FP32 band solves of up to two tiles of half-bandwidth (the local
solves of 2D boxes) at each depth of their tile ring: two turns ahead, one turn
ahead for long strips whose vector leaves no room for two and for batches of more
problems than SMs with a wide far tile, and the solve without a ring beyond.

Reference: a chosen solution, the right-hand side formed from it in FP64 by the
diagonals; diagonally dominant matrices (off-diagonal row sums at most 1 against a
diagonal of at least 2, condition below 3): relative error <= 1e-4, the FP32 bound
of the band solves at tile edges.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402


# two turns; one turn (strips of each number of far boxes); no ring; more problems than SMs, wide and narrow
@pytest.mark.parametrize("count,n,bw", [
    (2, 20000, 64), (1, 33001, 64), (1, 36000, 50), (1, 38500, 38), (1, 40000, 30), (1, 43000, 64),
    (153, 300, 64), (320, 257, 57), (160, 300, 40), (400, 65, 31)])
def test_one_column_solve_at_each_ring_depth(count, n, bw):
    gen = torch.Generator(device="cuda").manual_seed(n)
    f64 = dict(device="cuda", dtype=torch.float64)
    A = torch.zeros((count, n, n), **f64)
    x = torch.randn((count, n), generator=gen, **f64)
    diag = 2.0 + torch.rand((count, n), generator=gen, **f64)
    A.diagonal(0, 1, 2).copy_(diag)
    b = diag * x
    for d in range(1, min(bw, n - 1) + 1):
        v = (torch.rand((count, n - d), generator=gen, **f64) - 0.5) / bw
        A.diagonal(-d, 1, 2).copy_(v)
        A.diagonal(d, 1, 2).copy_(v)
        b[:, d:] += v * x[:, :-d]
        b[:, :-d] += v * x[:, d:]
    bb = pkg.BandBatch(A, [n] * count, bw, precision=1)
    y = bb.solve(b[:, :, None].contiguous())[:, :, 0]
    err = ((y - x).norm(dim=1) / x.norm(dim=1)).max().item()
    assert err <= 1e-4, err
    bb.close()

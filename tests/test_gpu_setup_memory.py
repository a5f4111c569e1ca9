"""Device memory of a set-up: the FP32 start phase needs none of its own, and the
fine eigensolver holds seven FP64 blocks with FP64 factors, six and an FP32 one with
FP32 factors.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402

N, PARTS, OVERLAP, NEV = 160, 5, 2, 8


def _kappa():
    gen = torch.Generator(device="cuda").manual_seed(3)
    return torch.exp(torch.randn(N * N, generator=gen, dtype=torch.float64, device="cuda"))


def _setup(precision, **kw):
    return pkg.Hierarchy((N, N), _kappa(), (PARTS, PARTS), OVERLAP, 2, (1, 1), NEV, 0.3, precision=precision, **kw)


def test_start_phase_takes_no_memory_of_its_own():
    held = {}
    for iters in (0, 20):
        pkg.msdd.release_cache()
        _setup(1, fp32_start_iters=iters).close()
        held[iters] = pkg.msdd.cached_bytes()      # every block of the set-up: none is reused within a call
    assert held[20] <= held[0], held


@pytest.mark.parametrize("precision", [0, 1])
def test_device_bytes_of_a_hierarchy(precision):
    size = 4 if precision else 8
    # node boxes of the subdomains (Dirichlet boxes are no larger), rounded to tile rows
    w = [min(N, k * (N // PARTS) + N // PARTS + OVERLAP) - max(0, k * (N // PARTS) - OVERLAP) + 1 for k in range(PARTS)]
    total = 0
    for x in w:
        for y in w:
            rows = -(-x * y // 32) * 32
            tiles = rows // 32 * (-(-(x + 1) // 32) + 1) * 1024
            block = (7 * 8 * 32 if precision == 0 else 6 * 8 * 32 + 4 * 12) * rows
            stencils = (2 * 8 + 4) * 9 * rows
            total += 2 * (tiles + rows) * size + block + stencils + x * y * NEV * 8 + rows * 8
    n0 = NEV * PARTS * PARTS
    total += (5 + 9) * 8 * (N + 1) ** 2 + 8 * N * N + 4 * 8 * n0 * n0
    H = _setup(precision)
    held = H.stats()["device_bytes"]
    H.close()
    assert 0.9 * total <= held <= 1.02 * total, (held, total)

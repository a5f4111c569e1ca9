"""The number of FP32 start iterations: one that the caller chose is run in full,
whatever the spectra need; under the default (20) a set-up whose subdomains all
converge sooner ends sooner.  Counted by the profiled intervals of the start
phase, two an iteration (the fine subdomains, 16 of them, are one group).
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2106_06404_gb300 as pkg  # noqa: E402


def _start_iterations(**kw):
    # a constant coefficient: few small eigenvalues and a large gap, ten or 13 iterations do
    k = torch.ones(64 * 64, dtype=torch.float64, device="cuda")
    H = pkg.Hierarchy((64, 64), k, (4, 4), 2, 2, (1, 1), 4, 0.3, precision=1, profile=1, **kw)
    n = H.stats()["prof"]["fine_gevp_fp32_start_other"]["launches"]
    H.close()
    return n / 2


@pytest.mark.parametrize("iters", [1, 5, 6, 7, 10, 11, 13, 14, 16, 19, 21, 30])
def test_chosen_number_of_start_iterations_is_run(iters):
    assert _start_iterations(fp32_start_iters=iters) == iters


def test_default_number_ends_early():
    assert 10 <= _start_iterations() < 20

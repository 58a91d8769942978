"""The untuned straight-line body is a fixed rule (amp_kernel.cu
gen_body_variant), so that the FP32 rounding of a small call does not depend on
how a build's kernels happen to spill: it is variant 1 (shared partials, 128
registers) of every process."""
import pytest

from paper_0909_5257_gb300 import phasespace as ps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pdg", [[21] * 4, [2, -2, 21, 21], [2, 2, 2, 2], [21] * 5, [2, -2, 21, 21, 21], [2, 2, 2, 2, 21]])
def test_untuned_body_is_the_first_variant(pdg):
    from paper_0909_5257_gb300 import mea
    n = 801
    mom = torch.empty((n, len(pdg), 4), dtype=torch.float64, device="cuda")
    mea.generate_phase_space(len(pdg) - 2, n, mom, seed=ps.SEED_BASE + 77)
    got = []
    for variant in (0, 1):
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        mea.Process(pdg, auto_tune=False, kernel_variant=variant).evaluate(mom, out)
        got.append(out)
    torch.cuda.synchronize()
    assert torch.equal(got[0], got[1])

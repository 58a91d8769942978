"""The phased kernel's written-out vertex functions (vertex_pinned.cuh) against
the per-lane kernel, bit for bit, over crossings that reach every one of them:
quark lines between initial and final legs, two lines, equal and different
flavours; FUSED units of one to four rounds."""
import pytest

from paper_0909_5257_gb300 import phasespace as ps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pdg", [
    [21, 21, 2, -2, 21, 21], [2, 21, 2, 21, 21, 21], [-2, 21, -2, 21, 21, 21], [2, -2, 1, -1, 21, 21],
    [2, 1, 2, 1, 21, 21], [21, 21, 2, -2, 2, -2], [2, 21, 2, 1, -1, 21], [21, -2, -2, 2, -2, 21],
    [21, 21, 2, -2, 21, 21, 21], [2, 21, 2, 1, -1, 21, 21]])
def test_crossings_have_the_per_lane_bits(pdg):
    from paper_0909_5257_gb300 import mea
    n = 257
    mom = torch.empty((n, len(pdg), 4), dtype=torch.float64, device="cuda")
    mea.generate_phase_space(len(pdg) - 2, n, mom, seed=ps.SEED_BASE + 79)
    got = []
    for mode in (0, 1):
        out, flag = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda")
        mea.Process(pdg, helicity_sharing=mode, auto_tune=False).evaluate(mom, out, flags=flag)
        got.append((out, flag))
    torch.cuda.synchronize()
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])

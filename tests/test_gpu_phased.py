"""The phased amplitude kernel (amp_phased_kernel.cu), the tensor-core path's
default, against the per-lane interpreter: the same operations on the same
inputs, so |M|^2 and the flags are the same bit for bit -- for one event, a few
(CTAs of the largest size), counts around the number of SMs, several chunks
with a ragged tail, and after autotuning (another CTA size)."""
import pytest

from paper_0909_5257_gb300 import phasespace as ps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    ("gg>gggg", [21] * 6, (300.0, 3000.0), (1, 151, 1037)),
    ("uu~>gggg", [2, -2] + [21] * 4, (300.0, 3000.0), (1, 305, 2111)),
    ("uu>uugg", [2, 2, 2, 2, 21, 21], (300.0, 3000.0), (7, 1201)),
    ("uu>uuggg", [2, 2, 2, 2, 21, 21, 21], (500.0, 5000.0), (1, 517)),
    ("ug>ugggg", [2, 21, 2, 21, 21, 21, 21], (500.0, 5000.0), (3, 203)),
    ("gg>ggggg", [21] * 7, (500.0, 5000.0), (1, 97)),
]


def _run(P, mom):
    from paper_0909_5257_gb300 import mea
    n = mom.shape[0]
    out = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    fl = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")
    P.evaluate(mom, out, precision=mea.PREC_MIXED, flags=fl)
    P.check_status()
    return out, fl


@pytest.mark.parametrize("name,pdg,rs,counts", CASES)
def test_phased_kernel_equals_per_lane_bit_for_bit(name, pdg, rs, counts):
    from paper_0909_5257_gb300 import mea
    n = max(counts)
    mom = torch.empty((n, len(pdg), 4), dtype=torch.float64, device="cuda")
    mea.generate_phase_space(len(pdg) - 2, n, mom, seed=ps.SEED_BASE + 717, rs_lo=rs[0], rs_hi=rs[1])
    a, fa = _run(mea.Process(pdg, helicity_sharing=1, auto_tune=False), mom)
    assert torch.isfinite(a).all()
    P = mea.Process(pdg, auto_tune=False)
    chunked = mea.Process(pdg, auto_tune=False, chunk_events=40)
    for k in counts:
        b, fb = _run(P, mom[:k])
        assert torch.equal(a[:k], b) and torch.equal(fa[:k], fb), k
    b, fb = _run(chunked, mom)
    assert torch.equal(a, b) and torch.equal(fa, fb)
    r = P.autotune(mom, torch.empty(n, dtype=torch.float64, device="cuda"), precision=mea.PREC_MIXED)
    assert r["helicity_shared"] == 3 and r["candidates"] >= 2, r
    b, fb = _run(P, mom)
    assert torch.equal(a, b) and torch.equal(fa, fb), r

"""The ordered recursion (ordered_kernel.cu), the FP64 path of the
non-vanishing helicity sum, against the per-lane kernels of the diagram program
(which the sum over all 2^n combinations runs): families, crossings, one event,
ragged counts, listed events (re-evaluation), the fixed-array entry point and
every tile of the autotuner."""
import pytest

from paper_0909_5257_gb300 import phasespace as ps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    ([21] * 4, (1, 4097)), ([21] * 5, (1, 1000)), ([21] * 6, (3, 307)), ([21] * 7, (5,)),
    ([2, -2, 21, 21], (1, 2049)), ([2, -2] + [21] * 3, (777,)), ([2, -2] + [21] * 4, (153,)), ([2, -2] + [21] * 5, (9,)),
    ([2, 2, 2, 2], (33,)), ([2, 2, 2, 2, 21], (1, 1025)), ([2, 2, 2, 2, 21, 21], (70,)), ([2, 2, 2, 2, 21, 21, 21], (5,)),
    ([2, 1, 2, 1, 21, 21, 21], (7,)), ([2, 21, 2, 21, 21], (100,)), ([2, -2, 2, -2, 21], (100,)), ([21, 2, 2, 21, 21, 21], (40,)),
]


@pytest.mark.parametrize("pdg,counts", CASES)
def test_ordered_recursion_equals_the_diagram_sum(pdg, counts):
    from paper_0909_5257_gb300 import mea
    n = max(counts)
    mom = torch.empty((n, len(pdg), 4), dtype=torch.float64, device="cuda")
    mea.generate_phase_space(len(pdg) - 2, n, mom, seed=ps.SEED_BASE + 911, rs_lo=300.0, rs_hi=3000.0)

    def run(P, k=n, hel_mode=0, prec=mea.PREC_FP64, noalloc=False):
        out = torch.full((k,), float("nan"), dtype=torch.float64, device="cuda")
        fl = torch.full((k,), 0xFF, dtype=torch.uint8, device="cuda")
        if noalloc:
            P.evaluate_noalloc(mom[:k], out, precision=prec, flags=fl)
        else:
            P.evaluate(mom[:k], out, precision=prec, flags=fl, hel_mode=hel_mode)
        torch.cuda.synchronize()
        return out, fl

    P = mea.Process(pdg, auto_tune=False)
    ref, fr = run(P, hel_mode=mea.HEL_SUM_ALL)
    got, fg = run(P)
    # two FP64 evaluations of the same sum, each pinned to the oracle at 1e-12 per event
    assert torch.allclose(got, ref, rtol=2e-12, atol=0), float((got / ref - 1).abs().max())
    assert torch.equal(fr, fg)
    for k in counts:
        part, _ = run(P, k)
        assert torch.equal(part, got[:k])
    fixed, _ = run(P, noalloc=True)
    assert torch.equal(fixed, got)
    # every event flagged: the mixed path's re-evaluation is this path
    every = mea.Process(pdg, flag_threshold=1e-30, auto_tune=False)
    mixed, fm = run(every, prec=mea.PREC_MIXED)
    assert torch.equal(mixed, got) and bool((fm & mea.FLAG_REEVALUATED).all())
    r = P.autotune(mom, torch.empty(n, dtype=torch.float64, device="cuda"), precision=mea.PREC_FP64)
    assert r["candidates"] >= 1
    tuned, _ = run(P)
    assert torch.equal(tuned, got), r

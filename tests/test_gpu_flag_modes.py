"""Amplitude-kernel choices (helicity_sharing 0 to 4) with the flag threshold near the
median indicator, so that events lie close to it on both sides.  Without
re-evaluation every mode gives the same |M|^2 bit for bit.  The indicator's sum of
magnitudes is added in another order by the phased kernel: a sum of K
non-negative FP32 terms is within K 2^-24 of the exact one in any order, so a mode's
flagged events are those of the threshold moved by twice that, at least and at
most, and events that two modes flag alike have the same bits."""
import pytest

from paper_0909_5257_gb300 import phasespace as ps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pdg,n,rs", [([21] * 6, 20000, (300.0, 3000.0)), ([2, -2] + [21] * 4, 40000, (300.0, 3000.0)),
                                      ([2, 2, 2, 2, 21, 21], 40000, (300.0, 3000.0)), ([2, -2] + [21] * 5, 4000, (500.0, 5000.0)),
                                      ([2, 2, 2, 2, 21, 21, 21], 6000, (500.0, 5000.0))])
def test_modes_agree_up_to_the_rounding_of_the_indicator(pdg, n, rs):
    from paper_0909_5257_gb300 import mea
    mom = torch.empty((n, len(pdg), 4), dtype=torch.float64, device="cuda")
    mea.generate_phase_space(len(pdg) - 2, n, mom, seed=ps.SEED_BASE + 404, rs_lo=rs[0], rs_hi=rs[1])

    def run(mode, threshold, reeval):
        P = mea.Process(pdg, helicity_sharing=mode, flag_threshold=threshold, reeval_fp64=reeval, auto_tune=False)
        out, flag = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda")
        P.evaluate(mom, out, flags=flag)
        P.check_status()
        return out, (flag & mea.FLAG_CANCEL) != 0, P.info["n_diagrams"]

    lo, hi = 32 * 2.0 ** -24, 1e-3  # the indicator is u (32 + kappa)
    for _ in range(40):
        mid = (lo * hi) ** 0.5
        if int(run(0, mid, False)[1].sum()) > n // 2:
            lo = mid
        else:
            hi = mid
    plain, flagged, diagrams = run(0, hi, False)
    assert n // 4 < int(flagged.sum()) < 3 * n // 4
    d = 2 * diagrams * 2.0 ** -24
    surely, possibly = run(0, hi * (1 + d), False)[1], run(0, hi * (1 - d), False)[1]
    first = run(0, hi, True)
    for mode in range(1, 5):
        try:
            out, f, _ = run(mode, hi, False)
        except mea.MeaError as e:
            assert e.status == -2, (mode, e)  # a layout that does not cover the process
            continue
        assert torch.equal(out, plain), mode
        assert not bool((surely & ~f).any()) and not bool((f & ~possibly).any()), mode
        out, f, _ = run(mode, hi, True)
        alike = f == first[1]
        assert torch.equal(out[alike], first[0][alike]), mode

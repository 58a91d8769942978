"""Flipped helicity combinations of pure-gluon processes (generator.h,
HelLanes): the sum over the non-vanishing combinations evaluates one of each
pair.  Evaluated one by one, a combination and its flipped one give the same
|M_h|^2 bit for bit, and the sum over all of them is the helicity sum."""
import pytest

from paper_0909_5257_gb300 import phasespace as ps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_final,n", [(2, 1), (2, 777), (3, 333), (4, 65)])
@pytest.mark.parametrize("prec", [0, 1])
def test_flipped_combinations_are_equal_and_sum_up(n_final, n, prec):
    from paper_0909_5257_gb300 import mea
    P = mea.Process([21] * (n_final + 2), auto_tune=False)
    mom = torch.empty((n, n_final + 2, 4), dtype=torch.float64, device="cuda")
    mea.generate_phase_space(n_final, n, mom, seed=ps.SEED_BASE + 311)
    total = torch.empty(n, dtype=torch.float64, device="cuda")
    P.evaluate(mom, total, precision=prec)
    hel = P.helicities()
    assert len(hel) % 2 == 0
    one = {}
    for row in hel:
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        given = torch.tensor(row, dtype=torch.int8, device="cuda").repeat(n, 1).contiguous()
        P.evaluate(mom, out, precision=prec, hel_mode=mea.HEL_GIVEN, hel=given)
        one[tuple(row)] = out
    for row in hel:
        assert torch.equal(one[tuple(row)], one[tuple(-row)])
    added = sum(one.values())
    # FP64: rounding of the sum; mixed: FP32 amplitudes, another colour path for 4 jets
    rtol = 1e-12 if prec == 0 else 2e-5
    assert torch.allclose(added, total, rtol=rtol, atol=0)

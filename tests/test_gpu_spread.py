"""Small calls of the straight-line kernels take smaller tiles (amp_kernel.cu,
gen_spread): every event has the bits it has in a call of full tiles, at counts
around one event per SM, ragged tiles and the first full tile."""
import pytest

from paper_0909_5257_gb300 import phasespace as ps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("pdg", [[21] * 4, [2, -2, 21, 21], [2, 2, 2, 2], [21] * 5, [2, -2, 21, 21, 21], [2, 2, 2, 2, 21]])
def test_small_calls_have_the_bits_of_a_large_one(pdg, precision):
    from paper_0909_5257_gb300 import mea
    prec = mea.PREC_MIXED if precision == "mixed" else mea.PREC_FP64
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N = 40000
    mom = torch.empty((N, len(pdg), 4), dtype=torch.float64, device="cuda")
    mea.generate_phase_space(len(pdg) - 2, N, mom, seed=ps.SEED_BASE + 78)
    P = mea.Process(pdg, auto_tune=False)
    ref, rflag = torch.empty(N, dtype=torch.float64, device="cuda"), torch.empty(N, dtype=torch.uint8, device="cuda")
    P.evaluate(mom, ref, precision=prec, flags=rflag)
    for n in (1, 2, sms - 1, sms, sms + 1, 777, 16 * sms, 21 * sms - 1, 25 * sms + 1, 85 * sms + 1):
        out, flag = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda")
        P.evaluate(mom[:n], out, precision=prec, flags=flag)
        torch.cuda.synchronize()
        assert torch.equal(out, ref[:n]) and torch.equal(flag, rflag[:n]), n

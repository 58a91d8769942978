"""Which kernels a process runs (mea_process_kernels): the recursion on the FP64 path
and the phased kernel on the mixed path are the ones that their comparisons with
other kernels compare, not a fallback."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# tests/test_gpu_ordered.py, tests/test_gpu_phased.py, tests/test_gpu_phased_crossings.py
RECURSION = [[21] * 5, [21] * 6, [21] * 7, [2, -2, 21, 21], [2, -2] + [21] * 3, [2, -2] + [21] * 4, [2, -2] + [21] * 5,
             [2, 2, 2, 2], [2, 2, 2, 2, 21], [2, 2, 2, 2, 21, 21], [2, 2, 2, 2, 21, 21, 21], [2, 1, 2, 1, 21, 21, 21],
             [2, 21, 2, 21, 21], [2, -2, 2, -2, 21], [21, 2, 2, 21, 21, 21]]
PHASED = [[21] * 6, [2, -2] + [21] * 4, [2, 2, 2, 2, 21, 21], [2, 2, 2, 2, 21, 21, 21], [2, 21, 2, 21, 21, 21, 21], [21] * 7,
          [21, 21, 2, -2, 21, 21], [2, 21, 2, 21, 21, 21], [-2, 21, -2, 21, 21, 21], [2, -2, 1, -1, 21, 21],
          [2, 1, 2, 1, 21, 21], [21, 21, 2, -2, 2, -2], [2, 21, 2, 1, -1, 21], [21, -2, -2, 2, -2, 21],
          [21, 21, 2, -2, 21, 21, 21], [2, 21, 2, 1, -1, 21, 21]]


@pytest.mark.parametrize("pdg", RECURSION)
def test_fp64_path_is_the_recursion(pdg):
    from paper_0909_5257_gb300 import mea
    assert mea.Process(pdg).kernels()["fp64_recursion"] == 1


@pytest.mark.parametrize("pdg", PHASED)
def test_mixed_path_is_phased(pdg):
    from paper_0909_5257_gb300 import mea
    k = mea.Process(pdg).kernels()
    assert k["mixed_path"] == 2 and k["amplitude_kernel"] == 3 and k["phased_flops_per_event"] > 0
    for mode, kernel in ((1, 0), (2, 1), (3, 2), (4, 0)):
        other = mea.Process(pdg, helicity_sharing=mode).kernels()
        assert other["amplitude_kernel"] == kernel and other["phased_flops_per_event"] == 0, mode


def test_other_paths_and_errors():
    from paper_0909_5257_gb300 import mea
    k = mea.Process([21] * 4).kernels()  # straight-line in both precisions
    assert (k["fp64_recursion"], k["mixed_path"], k["amplitude_kernel"]) == (0, 0, -1)
    assert k["helicity_lanes"] == mea.Process([21] * 4).info["n_hel_nonzero"] // 2
    assert mea.Process([2, 21, 2, 21, 21]).kernels()["mixed_path"] == 2
    assert mea.Process([2, 21, 2, 21, 21], colour_mode=1).kernels()["mixed_path"] == 1
    with pytest.raises(mea.MeaError) as e:
        mea.Process([21] * 5, host_only=True).kernels()
    assert e.value.status == -2

"""rp_stats.step_bytes counts the singlet slices of a launch over all items only where they
go to device memory (twice: out and back in), and each launch once."""
import numpy as np
import pytest

from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# two_I, anisotropic, precision, whether the slices leave the chip
CASES = [([1] * 4, False, "fp64", False), ([1, 2, 1, 1], False, "fp32", False),
         ([1] * 6 + [2], True, "fp64", False), ([1, 2, 1, 2, 1, 2, 1, 1], False, "fp32", True),
         ([1] * 9 + [2, 2], False, "fp32", True)]


def _system(two_I, aniso=False):
    from paper_1612_09517_gb300 import rp
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    rp.use_torch_allocator()
    gen = wl.random_anisotropic if aniso else wl.random_isotropic
    n1 = (len(two_I) + 1) // 2
    return rp, rp.System(gen(n1, len(two_I) - n1, two_I=two_I, k_S=2.0, k_T=0.5, seed=3))


@pytest.mark.parametrize("profile", [0, 1])
@pytest.mark.parametrize("two_I,aniso,prec,off_chip", CASES)
def test_bytes_of_one_launch(two_I, aniso, prec, off_chip, profile):
    rp, sy = _system(two_I, aniso)
    st = sy.yields([1.0, 4.0], 3, 5, 0.3, precision=prec, profile=profile)["stats"]
    assert st["step_launches"] == 1
    # row_terms = n_cheb per propagation and macro-step
    want = 2.0 * st["row_terms"] * sy.Z * 2 * (8 if prec == "fp64" else 4) if off_chip else 0.0
    assert st["step_bytes"] == pytest.approx(want, rel=1e-12, abs=0)


def test_rounds_of_a_converged_call_count_once():
    rp, sy = _system([1, 2, 1, 2, 1, 2, 1, 1])
    r = [rp.rp_yields_converged(sy.handle, [1.0, 4.0], 1e-3, 4, 60, 5, 0.3,
                                rp.rp_default_options(profile=p)) for p in (0, 1)]
    assert r[0]["stats"]["step_launches"] > 1 and np.all(r[0]["M_used"] == r[1]["M_used"])
    assert r[0]["stats"]["step_bytes"] == pytest.approx(r[1]["stats"]["step_bytes"], rel=1e-12)

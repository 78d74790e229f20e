"""max_rows bounds the propagations kept in device memory; a launch over all items keeps
none, so it takes the CTAs that run at once whatever the bound."""
import numpy as np
import pytest

from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# two_I, anisotropic, kernel, precision, rows in flight of 32 propagations under max_rows = 2
CASES = [([1, 2, 1, 2, 1, 2, 1, 1], False, 0, "fp32", 32), ([1] * 7, False, 0, "fp64", 32),
         ([1] * 6 + [2], True, 0, "fp64", 32), ([1] * 5, False, 5, "fp32", 32),
         ([1] * 6, False, 0, "fp32", 2), ([1] * 9 + [2, 2], False, 0, "fp32", 2)]


@pytest.mark.parametrize("two_I,aniso,kernel,prec,rows", CASES)
def test_rows_in_flight(two_I, aniso, kernel, prec, rows):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    gen = wl.random_anisotropic if aniso else wl.random_isotropic
    n1 = (len(two_I) + 1) // 2
    sy = rp.System(gen(n1, len(two_I) - n1, two_I=two_I, k_S=2.0, k_T=0.5, seed=3))
    F, M, T = [0.0, 4.0], 16, 0.1
    r = [sy.yields(F, M, 5, T, per_sample=True, precision=prec, kernel=kernel, max_rows=m) for m in (0, 2)]
    assert r[1]["stats"]["rows"] == rows
    tol = 1e-10 if prec == "fp64" else 1e-5
    assert np.max(np.abs(r[0]["per_sample"] - r[1]["per_sample"])) < tol

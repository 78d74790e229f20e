"""The FP64 time integral of rows with few configurations, at and around its 32 lanes, its
32 columns and its largest size, 96 (a loose tolerance takes longer steps and more columns), and the
allocation-free entry that runs it with the per-term step kernel: every sample against the
on-chip kernels (1e-10)."""
import numpy as np
import pytest

from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = {1: [], 2: [1], 30: [2, 9], 32: [1] * 5, 36: [2, 2, 3], 64: [1] * 6, 96: [1, 2, 1, 1, 1, 1],
         125: [4, 4, 4], 128: [1] * 7}


@pytest.mark.parametrize("tol", [0.0, 1e-4])
@pytest.mark.parametrize("Z", list(CASES))
def test_few_configurations(Z, tol):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    two_I = CASES[Z]
    n1 = (len(two_I) + 1) // 2
    sy = rp.System(wl.random_isotropic(n1, len(two_I) - n1, two_I=two_I, k_S=2.0, k_T=0.5, J=0.1, seed=61)
                   if two_I else wl.SpinSystem([], [], np.zeros((0, 3, 3)), 2.0, 0.5, 0.1))
    assert sy.Z == Z
    F, M, T = [0.0, 4.0], 5, 0.3
    ref = sy.yields(F, M, 8, T, per_sample=True, precision="fp64", tol=tol)["per_sample"]
    got = [sy.yields(F, M, 8, T, per_sample=True, precision="fp64", tol=tol, kernel=1)["per_sample"],
           rp.rp_yields_static(sy.handle, F, M, 8, T, rp.rp_default_options(precision="fp64", tol=tol),
                               per_sample=True)["per_sample"]]
    for g in got:
        assert np.max(np.abs(g - ref)) < 1e-10

"""The low-rank time integral (weights planned on the device) at the edges of its
range: few and many Chebyshev terms, loose tolerances (a larger rank), strong
decay within one macro-step, configuration counts around a block's tile.

Tolerances are those of the yields: 1e-10 relative in FP64, 1e-5 in FP32."""
import math

import numpy as np
import pytest

from oracle import coherent, dense
from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = {"fp64": 1e-10, "fp32": 1e-5}


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    yield


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kernel", [1, 2, 5])
@pytest.mark.parametrize("n_cheb", [12, 32, 84, 88])
def test_terms_and_kernels_match_oracle(n_cheb, kernel, prec):
    from paper_1612_09517_gb300 import rp
    s = wl.random_isotropic(2, 2, two_I=[1, 2, 1, 1], k_S=1.0, k_T=3.0, J=0.2, seed=7)  # Z = 24
    r = rp.System(s).yields([0.0, 6.0], 3, 5, 0.3, per_sample=True, precision=prec, n_cheb=n_cheb,
                            kernel=kernel)
    psi0 = coherent.sample_states(s, 5, range(3))
    for i, B in enumerate([0.0, 6.0]):
        phS, _, _ = dense.sample_yields(s, B, 0.3, psi0)
        assert np.max(np.abs(r["per_sample"][i, :, 0] - phS) / phS) < TOL[prec]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_strong_decay_within_one_step(prec):
    """No nuclei at zero field: one macro-step with kbar h = 30; phi_S = 1 - exp(-k_S T)."""
    from paper_1612_09517_gb300 import rp
    sy = rp.System(wl.SpinSystem([], [], np.zeros((0, 3, 3)), 30.0, 30.0, 0.0))
    r = sy.yields([0.0], 2, 0, 1.0, precision=prec)
    assert abs(r["out"][0, 0] - (1.0 - math.exp(-30.0))) < TOL[prec]


@pytest.mark.parametrize("two_I", [[1] * 7, [1] * 7 + [2], [1] * 8 + [4]])
def test_tiles_and_loose_tolerance(two_I):
    """Z = 128, 384 and 1280 (one thread's two configurations, a partial tile, several tiles), and a
    tolerance of 1e-4, whose longer steps need more columns than one block of the factor: both
    precisions run the same plan, so they differ by FP32 rounding only."""
    from paper_1612_09517_gb300 import rp
    s = wl.random_isotropic(4, len(two_I) - 4, two_I=two_I, k_S=2.0, k_T=0.5, J=0.1, seed=48)
    sy = rp.System(s)
    kw = dict(per_sample=True, kernel=1, tol=1e-4)
    a = sy.yields([0.0, 4.0], 3, 8, 0.3, precision="fp64", **kw)["per_sample"]
    b = sy.yields([0.0, 4.0], 3, 8, 0.3, precision="fp32", **kw)["per_sample"]
    assert np.max(np.abs(a[..., 0] - b[..., 0]) / a[..., 0]) < TOL["fp32"]
    c = sy.yields([0.0, 4.0], 3, 8, 0.3, precision="fp64", per_sample=True, kernel=1)["per_sample"]
    assert np.max(np.abs(a[..., 0] - c[..., 0]) / c[..., 0]) < 1e-2

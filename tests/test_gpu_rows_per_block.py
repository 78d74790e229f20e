"""Several propagations in one block: small systems with so many propagations that a
thread takes whole configurations (k_chip_items with up to 32 rows per block), counts that
do not fill the last block, and batches whose smaller system runs in a block sized for the
larger one.  Every sample against the per-term kernels, 1e-10 (FP64) and 1e-5 (FP32)."""
import numpy as np
import pytest

from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = {"fp64": 1e-10, "fp32": 1e-5}
FIELDS, T, SEED = [0.0, 4.0], 0.1, 23

# two_I of the nuclei and samples per field: 2 M Z > 39064 takes the kernel
CASES = {"z1": ([], 20011), "z2": ([1], 10013), "z3": ([2], 6607), "z6": ([1, 2], 3313),
         "z16": ([1] * 4, 1249), "z24": ([1, 1, 5], 839), "z96": ([1, 2, 1, 1, 1, 1], 211)}


def _system(two_I, seed):
    n1 = (len(two_I) + 1) // 2
    if not two_I:
        return wl.SpinSystem([], [], np.zeros((0, 3, 3)), 3.0, 1.0, 0.2)
    return wl.random_isotropic(n1, len(two_I) - n1, two_I=two_I, k_S=3.0, k_T=1.0, J=0.2, seed=seed)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    yield


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name", list(CASES))
def test_every_row_of_a_block(name, prec):
    from paper_1612_09517_gb300 import rp
    two_I, M = CASES[name]
    sy = rp.System(_system(two_I, 41))
    a, b = (sy.yields(FIELDS, M, SEED, T, per_sample=True, precision=prec, kernel=k)["per_sample"]
            for k in (0, 1))
    assert np.max(np.abs(a[..., 0] - b[..., 0]) / np.maximum(b[..., 0], 1e-3)) < TOL[prec]
    assert np.max(np.abs(a[..., 1:] - b[..., 1:])) < TOL[prec]
    if not two_I:  # a singlet without nuclei stays one: phi_S = 1 - exp(-k_S T)
        assert np.max(np.abs(a[..., 0] - (1.0 - np.exp(-3.0 * T)))) < TOL[prec]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_smaller_system_in_a_larger_block(prec):
    from paper_1612_09517_gb300 import rp
    shapes, M = [[1, 1, 1, 2], [1] * 4], 701
    sy = [rp.System(_system(t, 43 + i)) for i, t in enumerate(shapes)]
    b = rp.rp_yields_batch(sy, [np.array(FIELDS)] * 2, [M] * 2, [T] * 2, SEED,
                           rp.rp_default_options(precision=prec))["out"]
    for i in range(2):
        one = sy[i].yields(FIELDS, M, SEED, T, precision=prec, pair_id=i, kernel=1)["out"]
        assert np.allclose(b[i], one, rtol=TOL[prec], atol=TOL[prec])

"""H psi of large systems: FP32 systems with at least eight spin-1/2 nuclei and a multiple of
256 configurations stage the partners of a block by bulk copies, the 20-spin-1/2 shape has
an instance of its own, the others read partners directly.  FP32 against the FP64 kernel
on the same vectors (1e-5 of the largest entry), and that one against the oracle."""
import numpy as np
import pytest

from oracle import spin
from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# outer spin-1/2, spin-1 and spin-3/2 nuclei beside the 256-configuration tile; just the
# tile; one nucleus short of it; the shape with an instance of its own
SHAPES = {"z6144": [1] * 9 + [2, 3], "z256": [1] * 8, "z1280": [1] * 8 + [4], "z384": [1] * 7 + [2],
          "z4608": [1] * 9 + [2, 2], "z2p20": [1] * 20}


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    yield


def _system(name, aniso):
    two_I = SHAPES[name]
    n1 = (len(two_I) + 1) // 2
    gen = wl.random_anisotropic if aniso else wl.random_isotropic
    return gen(n1, len(two_I) - n1, two_I=two_I, k_S=2.0, k_T=0.5, J=0.2, seed=47)


@pytest.mark.parametrize("B", [0.0, 4.0])
@pytest.mark.parametrize("aniso", [False, True])
@pytest.mark.parametrize("name", list(SHAPES))
def test_apply_h(name, aniso, B):
    from paper_1612_09517_gb300 import rp
    s = _system(name, aniso)
    sy = rp.System(s)
    n = 2 if sy.Z > 10000 else 3
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(n, sy.Z, 4, 2, generator=g, device="cuda", dtype=torch.float32)
    xd = x.double()
    y, yd = torch.empty_like(x), torch.empty_like(xd)
    rp.rp_apply_h(sy.handle, B, rp.RP_FP32, n, x.data_ptr(), y.data_ptr())
    rp.rp_apply_h(sy.handle, B, rp.RP_FP64, n, xd.data_ptr(), yd.data_ptr())
    assert (y.double() - yd).abs().max().item() < 1e-5 * yd.abs().max().item()
    if sy.Z <= 384:
        Heff = spin.hamiltonian(s, B) - 1j * spin.haberkorn(s)
        v, w = (sy.to_input_order(torch.view_as_complex(a).cpu().numpy().reshape(n, -1)) for a in (xd, yd))
        ref = v @ Heff.T
        assert np.max(np.abs(w - ref)) < 1e-13 * np.max(np.abs(ref))


def test_kernel_3_is_one_launch_per_term():
    from paper_1612_09517_gb300 import rp
    st = rp.System(_system("z6144", False)).yields([1.0], 2, 8, 0.1, kernel=3)["stats"]
    assert st["kernel_path"] == 1

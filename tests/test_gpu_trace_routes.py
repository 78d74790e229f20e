"""Time traces, electron observables and traces over basis states in every layout of a
propagation: one thread per configuration and state, several configurations per thread,
clusters of 2, 4 and 8 blocks, isotropic and anisotropic; against one launch per term
(1e-10 in FP64, 1e-5 in FP32)."""
import numpy as np
import pytest

from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = {"fp64": 1e-10, "fp32": 1e-5}
B, T, SEED = 4.0, 0.2, 19
# two_I of the nuclei; several configurations per thread from z600 on, clusters from z2304 on
ISO = {"z96": [1, 2, 1, 1, 1, 1], "z600": [1, 4, 1, 4, 2, 1], "z972": [2, 1, 2, 2, 1, 2, 2],
       "z2304": [1] * 8 + [2, 2], "z4608": [1] * 9 + [2, 2], "z9216": [1] * 10 + [2, 2],
       "z13824": [1] * 9 + [2] * 3}
ANISO = {"z48": [1] * 4 + [2], "z192": [1] * 6 + [2], "z768": [1] * 8 + [2], "z1536": [1] * 9 + [2]}
ALL = [(k, False) for k in ISO] + [(k, True) for k in ANISO]


def _system(name, aniso):
    from paper_1612_09517_gb300 import rp
    two_I = (ANISO if aniso else ISO)[name]
    n1 = (len(two_I) + 1) // 2
    gen = wl.random_anisotropic if aniso else wl.random_isotropic
    return rp.System(gen(n1, len(two_I) - n1, two_I=two_I, k_S=3.0, k_T=1.0, J=0.2, seed=83))


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    yield


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name,aniso", ALL)
def test_traces(name, aniso, prec):
    from paper_1612_09517_gb300 import rp
    sy = _system(name, aniso)
    rng = np.random.default_rng(3)
    A = rng.normal(size=(4, 4)) + 1j * rng.normal(size=(4, 4))
    for M in (1, 3):
        r = []
        for k in (0, 1):
            o = rp.rp_default_options(precision=prec, kernel=k)
            t, p = rp.rp_time_trace(sy.handle, B, M, SEED, T, o)
            r.append((t, p, rp.rp_time_observable(sy.handle, B, M, SEED, T, A, o)[1]))
        assert np.array_equal(r[0][0], r[1][0]) and r[0][0].size >= 3
        assert np.max(np.abs(r[0][1] - r[1][1])) < TOL[prec]
        assert np.max(np.abs(r[0][2] - r[1][2])) < TOL[prec] * np.abs(A).sum()


@pytest.mark.parametrize("det", [1, 2, 3])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name,aniso", [(n, False) for n in ISO if n not in ("z9216", "z13824")] +
                         [("z192", True), ("z768", True)])
def test_basis_states(name, aniso, prec, det):
    if aniso and det == 3:
        pytest.skip("J_z sectors are those of isotropic systems")
    sy = _system(name, aniso)
    kw = dict(per_sample=True, precision=prec, deterministic=det)
    a, b = (sy.yields([B], 5, SEED, 0.02, kernel=k, **kw) for k in (0, 1))
    assert np.max(np.abs(a["per_sample"] - b["per_sample"])) < TOL[prec]
    assert np.allclose(a["out"][:, :1], b["out"][:, :1], rtol=TOL[prec], atol=0)

"""Two calls with the same arguments give the same bits: per-sample yields of systems of up
to 1024 configurations in every kernel that takes them, of larger ones on clusters, and the
time trace of one sample.  Sums over threads, blocks and macro-steps run in a fixed order."""
import numpy as np
import pytest

from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FIELDS, T, SEED, CALLS = [0.5, 4.0], 0.6, 29, 6
ISO = {"z24": [1, 1, 5], "z96": [1, 2, 1, 1, 1, 1], "z256": [1] * 8, "z864": [1, 2] * 3 + [1, 1],
       "z2304": [1] * 8 + [2, 2], "z4608": [1] * 9 + [2, 2]}
ANISO = {"z24": [1, 5, 1], "z192": [1] * 6 + [2], "z768": [1, 1, 2] + [1] * 6}


def _system(two_I, aniso):
    from paper_1612_09517_gb300 import rp
    n1 = (len(two_I) + 1) // 2
    gen = wl.random_anisotropic if aniso else wl.random_isotropic
    return rp.System(gen(n1, len(two_I) - n1, two_I=two_I, k_S=3.0, k_T=1.0, J=0.2, seed=31))


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    yield


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name,aniso,kw",
                         [(n, False, {}) for n in ISO if n != "z4608"] +
                         [(n, True, {}) for n in ANISO] +
                         [("z864", False, dict(kernel=2)), ("z864", False, dict(graph=1)),
                          ("z768", True, dict(kernel=2)), ("z768", True, dict(kernel=5)),
                          ("z96", False, dict(M=300)), ("z4608", False, {})])
def test_same_bits(name, aniso, prec, kw):
    kw = dict(kw)
    M = kw.pop("M", 24)
    if prec == "fp64" and name in ("z2304", "z4608"):
        pytest.skip("one launch per term: sums of blocks, in any order")
    sy = _system((ANISO if aniso else ISO)[name], aniso)
    first = sy.yields(FIELDS, M, SEED, T, per_sample=True, precision=prec, **kw)
    for _ in range(CALLS):
        again = sy.yields(FIELDS, M, SEED, T, per_sample=True, precision=prec, **kw)
        assert np.array_equal(again["per_sample"], first["per_sample"])
        assert np.array_equal(again["out"], first["out"])


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name,aniso", [("z96", False), ("z864", False), ("z4608", False),
                                        ("z192", True)])
def test_same_bits_of_a_trace(name, aniso, prec):
    from paper_1612_09517_gb300 import rp
    sy = _system((ANISO if aniso else ISO)[name], aniso)
    first = rp.rp_time_trace(sy.handle, 4.0, 1, SEED, T, rp.rp_default_options(precision=prec))[1]
    for _ in range(CALLS):
        again = rp.rp_time_trace(sy.handle, 4.0, 1, SEED, T, rp.rp_default_options(precision=prec))[1]
        assert np.array_equal(again, first)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_same_bits_of_the_static_entry(prec):
    from paper_1612_09517_gb300 import rp
    sy = _system(ISO["z256"], False)
    o = rp.rp_default_options(precision=prec)
    first = rp.rp_yields_static(sy.handle, FIELDS, 8, SEED, T, o, per_sample=True)["per_sample"]
    for _ in range(CALLS):
        again = rp.rp_yields_static(sy.handle, FIELDS, 8, SEED, T, o, per_sample=True)["per_sample"]
        assert np.array_equal(again, first)

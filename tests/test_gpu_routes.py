"""Every way a propagation can be laid out on the chip, at the edges of its range:
one thread per configuration and electron state (few configurations), several
configurations per thread (more), clusters of 2, 4 and 8 blocks (beyond one block),
per-term kernels over global memory; isotropic and anisotropic, spins above 1, no
spin-1/2 nucleus at all, rows that do not fill a block.

Per-sample yields against the FP64 oracle, tolerances 1e-10 (FP64) and 1e-5 (FP32)."""
import functools

import numpy as np
import pytest

from oracle import chebyshev, coherent, dense
from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = {"fp64": 1e-10, "fp32": 1e-5}
FIELDS, T, SEED = [0.0, 4.0], 0.1, 17

# two_I of the nuclei; the first half of them on radical 1
ISO = {
    "z3": [2], "z20": [4, 3], "z24": [1, 1, 5], "z96": [1, 2, 1, 1, 1, 1],
    "z192": [1] * 6 + [2], "z256": [1] * 8, "z600": [1, 4, 1, 4, 2, 1],
    "z972": [2, 1, 2, 2, 1, 2, 2], "z1280": [1] * 8 + [4], "z2304": [1] * 8 + [2, 2],
    "z4608": [1] * 9 + [2, 2], "z10368": [1] * 7 + [2] * 4,
    "z8192": [1] * 13, "z15360": [1] * 10 + [4, 2],
}
ANISO = {
    "z1x3": [2], "z20": [4, 3], "z24": [1, 5, 1], "z96": [1, 2, 1, 1, 1, 1],
    "z192": [1] * 6 + [2], "z256": [1] * 8, "z768": [1, 1, 2] + [1] * 6, "z1536": [1] * 9 + [2],
    "z2560": [1] * 9 + [4], "z4096": [1] * 12, "z6144": [1] * 11 + [2],
}


@functools.lru_cache(maxsize=None)
def _system(name, aniso):
    two_I = (ANISO if aniso else ISO)[name]
    n1 = (len(two_I) + 1) // 2
    gen = wl.random_anisotropic if aniso else wl.random_isotropic
    return gen(n1, len(two_I) - n1, two_I=two_I, k_S=3.0, k_T=1.0, J=0.2, seed=71 + len(two_I))


@functools.lru_cache(maxsize=None)
def _oracle(name, aniso):
    """phi_S, phi_T and survival of sample 1 at FIELDS[1]."""
    s = _system(name, aniso)
    return chebyshev.propagate_yields(s, FIELDS[1], T, coherent.sample_states(s, SEED, [1])[0])


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    yield


def _check(got, o, prec):
    assert abs(got[0] - o[0]) < TOL[prec] * o[0]
    assert abs(got[1] - o[1]) < TOL[prec] * max(o[0], o[1])
    assert abs(got[2] - o[2]) < TOL[prec]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name,aniso", [(k, False) for k in ISO] + [(k, True) for k in ANISO])
def test_routes_match_oracle(name, aniso, prec):
    from paper_1612_09517_gb300 import rp
    sy = rp.System(_system(name, aniso))
    o = _oracle(name, aniso)
    for M in (3, 160):  # rows that leave the chip idle (split further) and rows that fill it
        if M == 160 and sy.Z > 2000:
            continue
        r = [sy.yields(FIELDS, M, SEED, T, per_sample=True, precision=prec, kernel=k)["per_sample"]
             for k in (0, 1)]
        for q in r:
            _check(q[1, 1], o, prec)
        # the two routes agree on every sample
        assert np.max(np.abs(r[0][..., 0] - r[1][..., 0]) / r[1][..., 0]) < TOL[prec]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("aniso", [False, True])
def test_uneven_batch_and_basis_states(aniso, prec):
    """Systems of different sizes share one launch; basis states start in the rotated frames."""
    from paper_1612_09517_gb300 import rp
    names = ["z20", "z24", "z96"]
    sy = [rp.System(_system(n, aniso)) for n in names]
    b = rp.rp_yields_batch(sy, [np.array(FIELDS)] * 3, [4] * 3, [T] * 3, SEED,
                           rp.rp_default_options(precision=prec))
    for i, n in enumerate(names):
        one = sy[i].yields(FIELDS, 4, SEED, T, precision=prec, pair_id=i)
        assert np.allclose(b["out"][i], one["out"], rtol=TOL[prec], atol=TOL[prec])
    s = _system("z24", aniso)
    tr = sy[1].yields([FIELDS[1]], 2, SEED, T, precision=prec, deterministic=1)
    assert abs(tr["out"][0, 0] - dense.trace_yields(s, FIELDS[1], T)[0]) < TOL[prec]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("aniso", [False, True])
def test_time_trace(aniso, prec):
    from paper_1612_09517_gb300 import rp
    s = _system("z24", aniso)
    sy = rp.System(s)
    t, out = rp.rp_time_trace(sy.handle, FIELDS[1], 3, SEED, 0.5, rp.rp_default_options(precision=prec))
    psi0 = coherent.sample_states(s, SEED, range(3))
    ps = np.mean([dense.singlet_probability(s, FIELDS[1], p, t) for p in psi0], axis=0)
    assert np.max(np.abs(out[:, 0] - ps)) < TOL[prec]

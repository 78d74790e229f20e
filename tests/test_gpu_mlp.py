"""The fused forward pass of the control-variate network at the edges of its tiles: widths
that fill a padded layer or not, one to three hidden layers, inputs of one to six weight
tiles, rows that do not fill a block, and a width beyond it (the layer-by-layer pass).

Tolerance 1e-5 of max(1, |g|), that of an FP32 forward pass of these depths."""
import numpy as np
import pytest

from oracle import mlp
from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("hidden,layers", [(1, 1), (64, 1), (65, 2), (128, 3), (200, 2), (256, 3),
                                           (257, 2)])
@pytest.mark.parametrize("n_nuc", [0, 2, 12, 24])
def test_forward_matches_reference(n_nuc, hidden, layers):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    n1 = (n_nuc + 1) // 2
    s = wl.random_isotropic(n1, n_nuc - n1, seed=3) if n_nuc else wl.SpinSystem(
        [], [], np.zeros((0, 3, 3)), 1.0, 1.0, 0.0)
    cv = rp.ControlVariate(rp.System(s), hidden=hidden, layers=layers)
    p = cv.get_params()
    w = torch.from_numpy(p).to(torch.bfloat16).float().numpy()  # forward weights are BF16
    o = 0
    ref_p = p.astype(np.float64)
    for r, c in mlp.shapes(cv.d_in, hidden, layers):
        ref_p[o:o + r * c] = w[o:o + r * c]
        o += r * c + r
    samples = np.arange(7, 7 + 133)  # one full block and five rows
    got = cv.eval(np.full(133, 3.0), samples, 1234)
    x = mlp.features(1234, 0, samples, s, 3.0, 10.0)
    ref, _ = mlp.forward(ref_p, x, cv.d_in, hidden, layers)
    assert np.max(np.abs(got - ref)) <= 1e-5 * max(1.0, np.max(np.abs(ref)))
    mu, vm = cv.mean([0.0, 3.0, 7.0], 200, 99)
    for i, B in enumerate([0.0, 3.0, 7.0]):
        g, _ = mlp.forward(ref_p, mlp.features(99, 0, np.arange(200), s, B, 10.0), cv.d_in, hidden,
                           layers)
        assert abs(mu[i] - g.mean()) <= 1e-5 * max(1.0, np.max(np.abs(g)))
        assert abs(vm[i] - g.var(ddof=1) / 200) <= 1e-4 * vm[i] + 1e-12

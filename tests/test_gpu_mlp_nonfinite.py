"""Activations of the fused forward pass that overflow, or that BF16 would round to infinity:
rows with an infinite activation give what FP32 multiply-adds give (an infinity or NaN),
rows with large finite ones stay finite, and neither touches the other rows of its block."""
import numpy as np
import pytest

from oracle import mlp
from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BIG = float(torch.tensor(3.3e38).to(torch.bfloat16))


def _forward(p, x, d_in, hidden, layers):
    """FP64 sums rounded to FP32 after every layer, BF16 weights."""
    o, a = 0, x
    with np.errstate(all="ignore"):
        for i, (r, c) in enumerate(mlp.shapes(d_in, hidden, layers)):
            W = torch.from_numpy(p[o:o + r * c].reshape(r, c)).to(torch.bfloat16).double().numpy()
            z = (a[:, None, :] * W[None]).sum(-1) + p[o + r * c:o + r * c + r].astype(np.float64)
            o += r * c + r
            a = z.astype(np.float32).astype(np.float64)
            if i < layers:
                a = (a / (1.0 + np.exp(-a))).astype(np.float32).astype(np.float64)
    return a[:, 0]


@pytest.mark.parametrize("hidden,layers,second", [(40, 2, "positive"), (40, 2, "mixed"), (256, 2, "positive"),
                                                  (256, 3, "mixed"), (64, 1, "positive")])
def test_infinities_and_large_values(hidden, layers, second):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    s = wl.config2().system
    cv = rp.ControlVariate(rp.System(s), hidden=hidden, layers=layers)
    rng = np.random.default_rng(hidden + layers)
    parts = []
    for i, (r, c) in enumerate(mlp.shapes(cv.d_in, hidden, layers)):
        W = rng.normal(size=(r, c)) / np.sqrt(c)
        if i == 0:  # unit 0: a large multiple of |b_1| + |b_2|, infinite for about half of the samples
            W[0] = 0.0
            W[0, 3 * s.n_nuc + 6:3 * s.n_nuc + 8] = BIG
        elif i == 1 and layers > 1:
            W[:, 0] = 1e-30 * rng.uniform(0.5, 1.0, r) * (1 if second == "positive" else rng.choice([-1, 1], r))
        if i == layers:  # the output layer
            W = np.abs(W) * (1e-30 if layers == 1 else 1.0)
        parts += [W.astype(np.float32).ravel(), (0.1 * rng.normal(size=r)).astype(np.float32)]
    p = np.concatenate(parts)
    cv.set_params(p)
    n = 300
    x = mlp.features(7, 0, np.arange(n), s, 3.0, 10.0).astype(np.float32).astype(np.float64)
    ref = _forward(p, x, cv.d_in, hidden, layers)
    got = cv.eval(np.full(n, 3.0), np.arange(n), 7)
    ok = np.isfinite(ref)
    assert 30 < ok.sum() < n - 30
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(got[~ok & ~np.isnan(ref)], ref[~ok & ~np.isnan(ref)])
    assert np.max(np.abs(got[ok] - ref[ok]) / np.abs(ref[ok])) < 1e-5

"""Rounding of the fused forward pass: no larger than that of the layer-by-layer pass in
rounded FP32, for single samples and, without a bias, for the mean and the variance.  The
layer-by-layer pass evaluates the same network, its hidden layers padded with zero units
beyond the fused pass's width; the reference is FP64 on the same features.

With n samples of rms error e the mean of unbiased errors is of the order of e / sqrt(n), that
of the relative variance twice that; the bounds are twice and eight times e / sqrt(n) above
the layer-by-layer pass's own, means over six networks."""
import numpy as np
import pytest

from oracle import mlp
from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

WIDE, N, B = 264, 4096, 5.0


def _pad(p, d_in, hidden, layers):
    out, o = [], 0
    for i, (r, c) in enumerate(mlp.shapes(d_in, hidden, layers)):
        W = np.zeros((r if i == layers else WIDE, c if i == 0 else WIDE), np.float32)
        b = np.zeros(W.shape[0], np.float32)
        W[:r, :c], b[:r] = p[o:o + r * c].reshape(r, c), p[o + r * c:o + r * c + r]
        o += r * c + r
        out += [W.ravel(), b]
    return np.concatenate(out)


def _forward64(p, x, d_in, hidden, layers):
    o, a = 0, torch.from_numpy(x).cuda()
    for i, (r, c) in enumerate(mlp.shapes(d_in, hidden, layers)):
        W = torch.from_numpy(p[o:o + r * c].reshape(r, c)).to(torch.bfloat16).double().cuda()
        a = a @ W.T + torch.from_numpy(p[o + r * c:o + r * c + r]).double().cuda()
        o += r * c + r
        if i < layers:
            a = a * torch.sigmoid(a)
    return a[:, 0].cpu().numpy()


@pytest.mark.parametrize("ratio", [50.0, 1e4])
@pytest.mark.parametrize("hidden,layers", [(256, 3), (64, 1)])
def test_inputs_of_different_magnitude(hidden, layers, ratio):
    """The field feature is `ratio` times the others, its weights as much smaller."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    s = wl.config2().system
    sy = rp.System(s)
    e = []
    for seed in range(4):
        fused = rp.ControlVariate(sy, hidden=hidden, layers=layers, init_seed=seed + 1)
        wide = rp.ControlVariate(sy, hidden=WIDE, layers=layers)
        p = fused.get_params()
        p[:hidden * fused.d_in].reshape(hidden, -1)[:, -1] /= ratio
        fused.set_params(p)
        wide.set_params(_pad(p, fused.d_in, hidden, layers))
        x = mlp.features(11, 0, np.arange(N), s, 10.0 * ratio, 10.0).astype(np.float32).astype(np.float64)
        ref = _forward64(p, x, fused.d_in, hidden, layers)
        e.append([np.sqrt(np.mean((cv.eval(np.full(N, 10.0 * ratio), np.arange(N), 11) - ref) ** 2))
                  for cv in (fused, wide)])
    rms_f, rms_w = np.mean(e, axis=0)
    assert rms_f <= rms_w


@pytest.mark.parametrize("hidden,layers", [(256, 3), (256, 1), (200, 2), (128, 3), (64, 2)])
def test_no_more_rounding_than_fp32(hidden, layers):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    rp.use_torch_allocator()
    s = wl.config2().system
    sy = rp.System(s)
    e = []
    for seed in range(6):
        fused = rp.ControlVariate(sy, hidden=hidden, layers=layers, init_seed=seed + 1)
        wide = rp.ControlVariate(sy, hidden=WIDE, layers=layers)
        p = fused.get_params()
        if seed >= 3:  # biases, and weights of another distribution
            rng = np.random.default_rng(seed)
            p = (p * rng.uniform(0.5, 2.0, p.size) + 0.1 * np.std(p) * rng.normal(size=p.size)).astype(np.float32)
            fused.set_params(p)
        wide.set_params(_pad(p, fused.d_in, hidden, layers))
        x = mlp.features(11 + seed, 0, np.arange(N), s, B, 10.0).astype(np.float32).astype(np.float64)
        ref = _forward64(p, x, fused.d_in, hidden, layers)
        scale = np.sqrt(np.mean(ref ** 2))
        row = []
        for cv in (fused, wide):
            d = cv.eval(np.full(N, B), np.arange(N), 11 + seed) - ref
            mu, vm = cv.mean([B], N, 11 + seed)
            row.append([np.sqrt(np.mean(d ** 2)) / scale, abs(mu[0] - ref.mean()) / scale,
                        abs(vm[0] / (ref.var(ddof=1) / N) - 1.0)])
        e.append(row)
    (rms_f, mu_f, var_f), (rms_w, mu_w, var_w) = np.mean(e, axis=0)
    assert rms_f <= rms_w
    assert mu_f <= mu_w + 2.0 * rms_w / np.sqrt(N)
    assert var_f <= var_w + 8.0 * rms_w / np.sqrt(N)

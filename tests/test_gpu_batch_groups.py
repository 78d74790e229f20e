"""Size groups of a batch that run beside each other: the same results as one system at a
time, also where the allocator cannot hold the scratch of all groups at once."""
import numpy as np
import pytest

from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# Z = 12 to 768 in FP64, to 4608 (clusters) in FP32: every group is one persistent launch
SHAPES = {"fp64": [[1, 2, 1], [1, 1, 1, 1, 2], [1] * 7 + [2], [1] * 8 + [2]],
          "fp32": [[1, 2, 1], [1] * 7 + [2], [1] * 8 + [2, 2], [1] * 9 + [2, 2]]}
FIELDS, T, M = np.array([0.0, 4.0]), 0.1, 6


@pytest.mark.parametrize("limited", [False, True])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_groups_match_single_systems(prec, limited):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    torch.cuda.set_device(0)
    from paper_1612_09517_gb300 import rp
    live, state = {}, {"now": 0, "peak": 0, "cap": 1 << 62, "refused": 0}

    def alloc(nbytes, stream, ctx):
        if state["now"] + nbytes > state["cap"]:
            state["refused"] += 1
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), 0, stream or 0)
        live[p] = int(nbytes)
        state["now"] += int(nbytes)
        state["peak"] = max(state["peak"], state["now"])
        return p

    def free(ptr, stream, ctx):
        state["now"] -= live.pop(ptr)
        torch.cuda.caching_allocator_delete(ptr)

    a, f = rp.ALLOC_FN(alloc), rp.FREE_FN(free)
    try:
        assert rp.LIB.rp_set_allocator(a, f, None) == 0
        sy = [rp.System(wl.random_isotropic((len(t) + 1) // 2, len(t) // 2, two_I=t, k_S=3.0, k_T=1.0,
                                            J=0.2, seed=90 + i)) for i, t in enumerate(SHAPES[prec])]
        opt = rp.rp_default_options(precision=prec)

        def batch():
            return rp.rp_yields_batch(sy, [FIELDS] * len(sy), [M] * len(sy), [T] * len(sy), 5, opt)["out"]

        one, alone = [], 0
        for i, s in enumerate(sy):
            state["peak"] = 0
            one.append(s.yields(FIELDS, M, 5, T, precision=prec, pair_id=i)["out"])
            alone = max(alone, state["peak"])
        state["peak"] = 0
        got = batch()
        if limited:
            assert state["peak"] > alone + (1 << 20), "the groups did not overlap"
            state["cap"] = state["peak"] - 1
            got = batch()
            assert state["refused"] > 0
        for i in range(len(sy)):
            # the same kernels on the same inputs; sums of FP64 atomics in another order
            assert np.allclose(got[i], one[i], rtol=1e-9, atol=1e-12)
    finally:
        rp.use_torch_allocator()
    assert state["now"] == 0 and not live

"""The cluster macro-steps integrate on a second stream from a second copy of the singlet
slices; where the allocator has no room for that copy they do without, with the same
results."""
import numpy as np
import pytest

from paper_1612_09517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("gram", [0, 1, 2])
def test_without_room_for_the_copy(gram):
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
        sy = rp.System(wl.config2().system)
        kw = dict(per_sample=True, precision="fp32", kernel=4, max_rows=4, gram=gram)
        one = sy.yields([0.0, 20.0], 4, 5, 0.05, **kw)["per_sample"]
        assert state["now"] == 0
        state["cap"] = state["peak"] - (16 << 20)  # the copy is 58 MB, what follows it is small
        two = sy.yields([0.0, 20.0], 4, 5, 0.05, **kw)["per_sample"]
        assert state["refused"] > 0
        # sums of FP64 atomics in another order
        assert np.allclose(one, two, rtol=1e-9, atol=1e-12)
    finally:
        rp.use_torch_allocator()
    assert state["now"] == 0 and not live

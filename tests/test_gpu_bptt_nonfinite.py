"""A training step is a function of its inputs alone: after a backward whose count
gradient held a NaN or an Inf (an overflowed loss scale, a bad batch), the next step
on clean inputs gives the bits of a context that never saw one.  Layer widths off
the operands' 64-column rows, in narrowing and widening order, so that each layer's
row padding lies where another one's values were."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("engine", ["tensor", "simt"])
@pytest.mark.parametrize("recompute", [False, True])
@pytest.mark.parametrize("sizes", [(70, 200, 20), (40, 130, 200, 33), (90, 33, 130, 10)])
def test_clean_step_after_a_nonfinite_one(sizes, recompute, engine, bad):
    from paper_2305_02510_gb300 import bptt
    batch, steps = 16, 30
    rng = np.random.default_rng(sum(sizes))
    x = torch.from_numpy((rng.random((steps, batch, sizes[0])) < 0.2).astype(np.uint8)).cuda()
    ws = [torch.from_numpy(rng.normal(0, np.sqrt(2.0 / a), (a, b)).astype(np.float32)).cuda().requires_grad_()
          for a, b in zip(sizes[:-1], sizes[1:])]
    ds = [rng.integers(1, 5, (a, b)).astype(np.uint8) for a, b in zip(sizes[:-1], sizes[1:])]
    gc = torch.from_numpy(rng.normal(0, 1, (batch, sizes[-1])).astype(np.float32)).cuda()
    poisoned = gc.clone()
    poisoned[3, 1] = bad

    def step(net, grad):
        counts = bptt.SNNFunction.apply(net, x, *ws)
        return [counts.detach(), *torch.autograd.grad(counts, ws, grad)]

    def net():
        return bptt.FFNet(sizes, ds, batch=batch, steps=steps, engine=engine, recompute=recompute)

    want = step(net(), gc)
    used = net()
    assert not all(bool(torch.isfinite(g).all()) for g in step(used, poisoned)[1:])
    for _ in range(2):
        for a, b in zip(step(used, gc), want):
            assert bool(torch.isfinite(a).all()) and torch.equal(a, b)

"""The tensor-core contractions at the edges of their tiles (one or two row tiles
a work item, ragged rows and columns, layers narrower than a tile) against the
CUDA-core engine.  The weights are multiples of 1/16 below 4 and the leak of
1/32, so every forward sum is exact in both engines: counts equal.  A gradient
carries the two-part BF16 split, at most 2^-16 of every product's factor, so its
Frobenius distance stays below 3 * 2^-16 per layer passed (three layers at most)
plus float32's own 1e-5."""

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


@pytest.mark.parametrize("recompute", [False, True])
@pytest.mark.parametrize("sizes,batch,steps", [
    ((70, 200, 130, 9), 72, 141),        # 80 row tiles x 2: two a work item, the last one ragged
    ((257, 129, 20), 128, 100),          # a second column tile of one column
    ((33, 129, 257), 8, 9),              # fewer rows than a tile
    ((16, 112, 16), 24, 11), ((64, 113, 1), 8, 20), ((1, 1, 1), 8, 3)])
def test_engines_agree(sizes, batch, steps, recompute):
    from paper_2305_02510_gb300 import bptt
    rng = np.random.default_rng(sum(sizes) + batch)
    x = torch.from_numpy((rng.random((steps, batch, sizes[0])) < 0.15).astype(np.uint8)).cuda()
    ws = [torch.from_numpy((np.round(rng.normal(0, 16 * np.sqrt(2.0 / a) + 1, (a, b))).clip(-63, 63) / 16)
                           .astype(np.float32)).cuda().requires_grad_() for a, b in zip(sizes[:-1], sizes[1:])]
    ds = [rng.integers(1, 5, (a, b)).astype(np.uint8) for a, b in zip(sizes[:-1], sizes[1:])]
    gc = torch.from_numpy(rng.normal(0, 1, (batch, sizes[-1])).astype(np.float32)).cuda()
    got = {}
    for engine in ("tensor", "simt"):
        net = bptt.FFNet(sizes, ds, batch=batch, steps=steps, leak=1.0 / 32, engine=engine, recompute=recompute)
        counts = bptt.SNNFunction.apply(net, x, *ws)
        got[engine] = (counts.detach(), torch.autograd.grad(counts, ws, gc))
    assert torch.equal(got["tensor"][0], got["simt"][0])
    bound = 3 * 3 * 2.0 ** -16 + 1e-5
    for a, b in zip(got["tensor"][1], got["simt"][1]):
        assert float((a.double() - b.double()).norm()) <= bound * float(b.double().norm())

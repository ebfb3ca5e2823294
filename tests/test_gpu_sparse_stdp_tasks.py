"""Sparse STDP at the edges of its tasks (a row or a column of a spiker, 128
synapses at a time): single-block and grid networks, rows and columns that are
empty, of one synapse, of 128 and of several times as many, more spikers in a
block than warps.  The weights and traces that a run leaves are recomputed from
the recorded spikes in float32, every product and sum rounded as the rule states
them: equal bit for bit."""

import numpy as np
import pytest

from paper_2305_02510_gb300 import sn as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("n,long_row,rate", [(40, 39, 0.3), (2048, 128, 0.1), (2049, 129, 0.02), (2100, 700, 0.3),
                                             (6001, 300, 0.05)])
def test_weights_follow_from_the_spikes(n, long_row, rate):
    rng = np.random.default_rng(n)
    steps = 40
    count = rng.integers(0, 12, n)
    count[::97] = long_row                  # a few long rows
    count[1::97] = 1
    pre = np.repeat(np.arange(n), count)
    post = (pre + 1 + rng.integers(0, n - 1, pre.size)) % n
    post[: n // 3] = np.where(pre[: n // 3] == 7, 8, 7)      # a long column
    key = np.unique(pre.astype(np.int64) * n + post)
    pre, post = (key // n).astype(np.int32), (key % n).astype(np.int32)
    w = rng.uniform(-0.5, 0.8, pre.size).astype(np.float32)
    f = lambda x: np.full(n, x, np.float32)
    ctx = S.sn_create(f(1.0), f(0.05), f(0.0), rng.integers(0, 3, n).astype(np.int32), pre, post, w,
                      np.ones(pre.size, np.int32), max_delay=1, record_steps=steps)
    S.sn_set_poisson(ctx, np.arange(n, dtype=np.int32), f(rate), f(1.3), 17)
    decay, ap, am, lo, hi = (np.float32(x) for x in (0.9, 0.03, 0.02, -0.6, 0.9))
    S.sn_stdp(ctx, decay, ap, am, lo, hi)
    for q in (1, 13, steps - 14):
        S.sn_run(ctx, q)
    spikes = S.unpack_raster(S.sn_get_spikes(ctx, 0, steps), n).astype(bool)
    assert spikes[5:].any(axis=1).all()
    x = np.zeros(n, np.float32)
    for s in spikes:
        up = ap * x[pre]
        row = (w + (np.where(s[post], up, np.float32(0)) - am * x[post])).clip(lo, hi)
        col = (w + up).clip(lo, hi)
        w = np.where(s[pre], row, np.where(s[post], col, w)).astype(np.float32)
        x = (decay * x + s.astype(np.float32)).astype(np.float32)
    assert np.array_equal(S.sn_get_weights(ctx).view(np.int32), w.view(np.int32))
    assert np.array_equal(S.sn_get_trace(ctx).view(np.int32), x.view(np.int32))

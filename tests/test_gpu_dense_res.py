"""Dense networks small enough for their weights to stay in shared memory: a run
in launches long enough for that form (4 steps, 12 with plasticity) leaves the
same spikes and the same saved state, byte for byte (voltages, refractory
counters, pending input, spike words, weights, traces), as the same run in launches of at most three steps, which
stream the rows from memory.  Sizes at the edges of a warp, of one block, of the
vector form (n % 4 == 0) and of the shared memory (the largest with and without
plasticity, and the first size past each, where both runs stream)."""

import numpy as np
import pytest

from paper_2305_02510_gb300 import sn as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

STEPS = 23


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()


def make(n, delay, stdp, slab):
    rng = np.random.default_rng(1000 * n + 10 * delay + stdp)
    w = rng.normal(0.0, 3.0 / np.sqrt(n + 8.0), (n, n)).astype(np.float32)
    np.fill_diagonal(w, 0.0)
    th = rng.uniform(0.7, 1.2, n).astype(np.float32)
    lk = rng.uniform(0.0, 0.1, n).astype(np.float32)
    ctx = S.sn_create_dense(th, lk, np.zeros(n, np.float32), rng.integers(0, 3, n).astype(np.int32), w, delay,
                            max_delay=4, flags=S.SN_DENSE_SLAB(slab) if slab else S.SN_AUTO, record_steps=STEPS)
    S.sn_set_poisson(ctx, np.arange(n, dtype=np.int32), np.full(n, 0.1, np.float32), np.full(n, 1.1, np.float32), 5)
    ne = 4 * STEPS
    S.sn_set_input(ctx, rng.integers(0, STEPS - 3, ne).astype(np.int32), rng.integers(0, n, ne).astype(np.int32),
                   rng.uniform(0.2, 1.5, ne).astype(np.float32))
    if stdp:
        S.sn_stdp(ctx, 0.9, 0.02, 0.015, -0.3, 0.3)
    return ctx


@pytest.mark.parametrize("n,slab", [(1, 0), (31, 0), (33, 0), (64, 0), (65, 0), (100, 0), (128, 0), (129, 0), (1000, 0),
                                    (1001, 0), (1001, 2), (700, 4), (701, 4), (1617, 0), (1618, 0), (1715, 0),
                                    (1716, 0)])
@pytest.mark.parametrize("stdp", [False, True])
def test_same_bytes_as_the_streaming_form(n, slab, stdp):
    delay = 1 if stdp or n % 2 else 3
    got, want = make(n, delay, stdp, slab), make(n, delay, stdp, slab)
    for q in (4, STEPS - 9, 1, 4):
        S.sn_run(got, q)
    for q in [3] * (STEPS // 3) + [1] * (STEPS % 3):
        S.sn_run(want, q)
    a = S.unpack_raster(S.sn_get_spikes(got, 0, STEPS), n)
    b = S.unpack_raster(S.sn_get_spikes(want, 0, STEPS), n)
    assert np.array_equal(a, b), f"raster differs first at step {int(np.nonzero((a != b).any(axis=1))[0][0])}"
    assert b[STEPS // 2:].any() or n == 1
    assert S.sn_get_counters(got) == S.sn_get_counters(want)
    assert S.sn_save(got) == S.sn_save(want)

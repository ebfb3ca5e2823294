"""Pull in blocks of three steps (networks of more than one block of threads):
every spike and state bit-identical to the oracle's mirror at the edges of the
kernel's ranges: the delays at which a neuron's spike word grows (8, 16, 32
bits: 12, 20, 36) and the lists above delay 3 begin, odd word counts, runs that
end anywhere in a block of steps, blocks of more than 672 threads, and a switch
to push and back in mid-run."""

import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_02510_gb300 import sn as S
from paper_2305_02510_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()


def network(seed, n, k, delays, integer, steps):
    """k incoming synapses a neuron, delays drawn from `delays`, events at about
    a hundredth of the neurons per step."""
    rng = np.random.default_rng(seed)
    post = np.repeat(np.arange(n, dtype=np.int32), k)
    pre = ((post + rng.integers(1, n, post.size)) % n).astype(np.int32)
    delay = rng.choice(np.asarray(delays), post.size).astype(np.int32)
    if integer:
        w, th, lk = rng.integers(-3, 7, post.size).astype(np.float64), np.full(n, 3.0), np.full(n, 1.0)
    else:
        w, th, lk = rng.normal(0.4, 0.4, post.size), rng.uniform(0.8, 1.2, n), rng.uniform(0.0, 0.1, n)
    wl = W._base(n, "i32" if integer else "f32", th, lk, np.zeros(n), rng.integers(0, 3, n).astype(np.int32),
                 int(max(delays)), steps)
    order = np.lexsort((post, pre))
    wl.update(pre=pre[order], post=post[order], weight=w[order], delay=delay[order])
    ne = max(20, n // 100) * steps
    val = rng.integers(5, 12, ne).astype(np.float64) if integer else rng.uniform(1.5, 3.0, ne)
    wl["events"] = dict(step=rng.integers(0, steps, ne).astype(np.int32),
                        neuron=rng.integers(0, n, ne).astype(np.int32), value=val)
    wl["name"] = f"pull-block-{seed}"
    return wl


def check(wl, runs, integer):
    steps = sum(runs)
    st, want, _ = O.run(wl, O.INT if integer else O.F32, steps)
    assert want[steps // 2:].sum() > 100
    ctx = S.from_workload(wl, flags=S.SN_PROP_PULL, record_steps=steps)
    for q in runs:
        S.sn_run(ctx, q)
    raster = S.unpack_raster(S.sn_get_spikes(ctx, 0, steps), wl["n"])
    v, r = S.sn_get_state(ctx)
    bad = np.nonzero((raster != want).any(axis=1))[0]
    assert bad.size == 0, f"raster differs first at step {int(bad[0])}"
    assert np.array_equal(np.asarray(v, np.float64), st.v) and np.array_equal(np.asarray(r), st.r)


@pytest.mark.parametrize("integer", [False, True])
@pytest.mark.parametrize("delays", [[1], [2, 3], [3], [4], [1, 4, 6, 7], range(1, 13), range(1, 14), range(1, 21),
                                    range(1, 22), [1, 36], range(30, 37), range(1, 38)])
def test_delays(delays, integer):
    delays = list(delays)
    wl = network(17 * max(delays) + len(delays), 2081, 9, delays, integer, 90)
    check(wl, [1, 2, 3, 4, 5, 6, 7, 62], integer)


@pytest.mark.parametrize("n", [1025, 1056, 4864, 4865, 9728, 30_001])
def test_sizes(n):
    check(network(n, n, 12, range(1, 17), False, 50), [50], False)


def test_wide_blocks():
    """More than 672 threads a block: 110,003 neurons, delays 1..12."""
    check(network(5, 110_003, 4, range(1, 13), False, 40), [7, 33], False)


def test_switch_in_mid_run():
    wl = network(23, 3001, 8, range(1, 10), True, 60)
    st, want, _ = O.run(wl, O.INT, 60)
    ctx = S.from_workload(wl, record_steps=60)
    for mode, q in ((S.SN_PUSH, 11), (S.SN_PULL, 8), (S.SN_PUSH, 5), (S.SN_PULL, 36)):
        S.sn_set_propagation(ctx, mode)
        S.sn_run(ctx, q)
    assert np.array_equal(S.unpack_raster(S.sn_get_spikes(ctx, 0, 60), wl["n"]), want)
    assert np.array_equal(np.asarray(S.sn_get_state(ctx)[0], np.float64), st.v)

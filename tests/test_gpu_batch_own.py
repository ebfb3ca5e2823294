"""Batched networks whose state stays in registers (every network of at most 1024
neurons, those on single warps at most 128): the same spikes and states, bit for
bit, as the general form, which the same networks take when one of 4096 neurons
joins them.  Sizes at the edges of a warp and of a thread's neurons, pending input
in shared and in global memory, runs of several lengths, and weights whose sums
reach both pieces of the fixed-point conversions (below and above 2^16)."""

import numpy as np
import pytest

from paper_2305_02510_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [1, 2, 31, 32, 33, 64, 96, 127, 128, 129, 255, 256, 257, 511, 513, 768, 1000, 1023, 1024]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()


def networks(integer):
    nets = []
    for k, n in enumerate(SIZES + SIZES[8:] + [4096]):
        wl = W.random_small(900 + k, n=n, integer=integer, steps=60, p=min(0.5, 20.0 / n), max_delay=1 + k % 8,
                            events_rate=1.5)
        wl["poisson"] = dict(neuron=np.arange(0, n, 3, dtype=np.int32), rate=np.full((n + 2) // 3, 0.08),
                             amplitude=np.full((n + 2) // 3, 9.0), seed=11)
        if not integer and k % 3 == 1:
            # sums from 2^-20 to beyond 2^20
            wl["weight"] = np.asarray(wl["weight"]) * np.exp2(np.random.default_rng(k).integers(-20, 21, len(wl["weight"])))
        nets.append(wl)
    return nets


def run(nets, config):
    from paper_2305_02510_gb300 import sn as S
    ctx = S.from_batch_workloads(nets, record_steps=60)
    S.sn_batch_config(ctx, *config)
    for q in (1, 37, 22):
        S.sn_run(ctx, q)
    S.sn_sync(ctx)
    v, r = S.sn_get_state(ctx)
    return S.split_batch_raster(S.sn_get_spikes(ctx, 0, 60), ctx.net_n), v, r


@pytest.mark.parametrize("config", [(0, 0), (0, 96 * 1024), (128, 80 * 1024), (128, 0)])
@pytest.mark.parametrize("integer", [False, True])
def test_same_bits_as_the_general_form(config, integer):
    nets = networks(integer)
    got, v, r = run(nets[:-1], config)
    want, v0, r0 = run(nets, config)
    assert sum(int(w[20:].sum()) for w in want[:-1]) > 1000
    for b, (x, y) in enumerate(zip(got, want)):
        assert np.array_equal(x, y), f"network {b} of {len(nets[b]['threshold'])} neurons"
    assert np.array_equal(np.asarray(v).view(np.int32), np.asarray(v0)[:len(v)].view(np.int32))
    assert np.array_equal(r, np.asarray(r0)[:len(r)])


def test_two_contexts_with_different_rings():
    """The shared-memory limit of the kernel is the process's: a second context
    with a smaller ring leaves the first one's graph launchable."""
    from paper_2305_02510_gb300 import sn as S
    nets = networks(True)[:6]
    a = S.from_batch_workloads(nets, record_steps=60)
    S.sn_batch_config(a, 0, 160 * 1024)
    S.sn_run(a, 10)
    b = S.from_batch_workloads(nets, record_steps=60)
    S.sn_batch_config(b, 0, 0)
    S.sn_run(b, 10)
    S.sn_run(a, 7)
    S.sn_run(b, 7)
    assert np.array_equal(S.sn_get_spikes(a, 0, 17), S.sn_get_spikes(b, 0, 17))

"""The pull store's forms on networks of many blocks: without a flag the order for
blocks of three steps, SN_PULL_PLAIN and SN_PULL_CODED the kernel that takes one step
at a time, and the same where the blocked kernel cannot count a list or hold a sum
(a region of more than 131,070 synapses; integer weights whose magnitudes reach 2^31).
Spikes and states equal the oracle's in every form."""

import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_02510_gb300 import sn as S
from paper_2305_02510_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FORMS = [0, S.SN_PULL_PLAIN, S.SN_PULL_CODED]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()


def plain_bytes(n, pre, post, delay, chunk):
    """Bytes of the plain store in two regions (delay >= 2, delay 1), as the one-step
    kernel reads it: within a block of `chunk` neurons by list length, then within 64
    by the delay-1 list, pairs padded to the longest list of 32."""
    long = np.bincount(post[delay >= 2], minlength=n)
    one = np.bincount(post[delay == 1], minlength=n)
    total = 0
    for b0 in range(0, n, chunk):
        order = b0 + np.argsort(-(long + one)[b0:b0 + chunk], kind="stable")
        for w0 in range(0, order.size, 64):
            part = order[w0:w0 + 64]
            part = part[np.argsort(-one[part], kind="stable")]
            for s0 in range(0, part.size, 32):
                q = part[s0:s0 + 32]
                total += ((int(long[q].max()) + 1) // 2 + (int(one[q].max()) + 1) // 2) * 32 * 16
    return total


def run(wl, form, steps):
    ctx = S.from_workload(wl, flags=S.SN_PROP_PULL | form, record_steps=steps)
    S.sn_run(ctx, steps)
    raster = S.unpack_raster(S.sn_get_spikes(ctx, 0, steps), wl["n"])
    v, r = S.sn_get_state(ctx)
    return S.sn_pull_store_info(ctx), raster, np.asarray(v, np.float64), np.asarray(r)


def check(wl, steps, mode, forms=FORMS):
    st, want, _ = O.run(wl, mode, steps)
    assert want.sum() > 100
    info = []
    for form in forms:
        i, raster, v, r = run(wl, form, steps)
        assert np.array_equal(raster, want) and np.array_equal(v, st.v) and np.array_equal(r, st.r), form
        info.append(i)
    return info


@pytest.mark.parametrize("integer", [False, True])
def test_flags_choose_the_kernel(integer):
    n, steps = 3000, 60
    wl = W.random_small(61, n=n, integer=integer, steps=steps, p=0.01, max_delay=9, events_rate=40.0)
    auto, plain, coded = check(wl, steps, O.INT if integer else O.F32)
    assert [i[0] for i in (auto, plain, coded)] == [S.SN_PULL_PLAIN, S.SN_PULL_PLAIN, S.SN_PULL_CODED]
    pre, post, delay = (np.asarray(wl[k]) for k in ("pre", "post", "delay"))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    chunk = (-(-n // 32) + sms - 1) // sms * 32
    assert plain[1] == plain_bytes(n, pre, post, delay, chunk) < auto[1]


def test_a_list_too_long_to_count():
    n, steps, m = 2000, 12, 131_072
    rng = np.random.default_rng(8)
    wl = W.random_small(62, n=n, integer=False, steps=steps, p=0.003, max_delay=5, events_rate=60.0)
    order = np.argsort(np.concatenate([wl["pre"], pre := rng.integers(0, n, m)]), kind="stable")
    add = dict(pre=pre, post=np.zeros(m), weight=rng.normal(0.0, 0.01, m), delay=np.full(m, 3))
    for k, x in add.items():
        wl[k] = np.concatenate([wl[k], x.astype(np.asarray(wl[k]).dtype)])[order]
    auto, plain = check(wl, steps, O.F32, FORMS[:2])
    assert auto == plain


@pytest.mark.parametrize("together", [False, True])
def test_integer_sums_past_32_bits(together):
    """200 synapses of 16,000,000 into neuron 0: a sum of 3.2e9 leaves int32, a fifth
    of it does not."""
    n, steps, k = 2000, 10, 200
    src = np.arange(100, 100 + k)
    wl = W._base(n, "i32", np.where(np.arange(n) == 0, 2.0 ** 23, 5.0), np.zeros(n), np.zeros(n),
                 np.zeros(n, np.int32), 4, steps)
    wl.update(pre=src.astype(np.int32), post=np.zeros(k, np.int32), weight=np.full(k, 16e6),
              delay=np.full(k, 4, np.int32), name="int-sums")
    fire = src if together else src[:40]
    wl["events"] = dict(step=np.repeat([1, 3, 4], fire.size).astype(np.int32),
                        neuron=np.tile(fire, 3).astype(np.int32), value=np.full(3 * fire.size, 9.0))
    if not together:
        auto, plain, _ = check(wl, steps, O.INT)
        assert auto == plain
        return
    for form in FORMS:
        ctx = S.from_workload(wl, flags=S.SN_PROP_PULL | form, record_steps=steps)
        S.sn_run(ctx, steps)
        with pytest.raises(S.SnError) as e:
            S.sn_sync(ctx)
        assert e.value.status == S.SN_EOVERFLOW


def drive(form, n, max_delay, integer):
    """Runs of one and a few steps, a reset after fewer and after more steps than there
    are row slots, a checkpoint taken back, weights replaced with spikes in flight, a
    push run in between: every raster and state along the way."""
    wl = W.random_small(63, n=n, integer=integer, steps=60, p=12.0 / n, max_delay=max_delay, events_rate=n / 60.0)
    ctx = S.from_workload(wl, flags=S.SN_PROP_PULL | form, record_steps=60)
    out = []

    def look(t0, t1):
        out.append(S.sn_get_spikes(ctx, t0, t1).copy())
        out.extend(np.asarray(x).copy() for x in S.sn_get_state(ctx))

    for runs in ((1, 1, 1), (5,), (1,) * 12 + (2, 3, 7, 1, 1), (30,)):
        S.sn_reset(ctx)
        for q in runs:
            S.sn_run(ctx, q)
        look(0, sum(runs))
    if not integer:
        S.sn_set_weights(ctx, np.asarray(wl["weight"], np.float32)[::-1].copy())
    S.sn_run(ctx, 4)
    look(30, 34)
    blob = S.sn_save(ctx)
    S.sn_run(ctx, 6)
    look(34, 40)
    S.sn_load(ctx, blob)
    S.sn_run(ctx, 1)
    S.sn_run(ctx, 5)
    look(34, 40)
    for mode, q in ((S.SN_PUSH, 3), (S.SN_PULL, 1), (S.SN_PULL, 4), (S.SN_PUSH, 1), (S.SN_PULL, 6)):
        S.sn_set_propagation(ctx, mode)
        S.sn_run(ctx, q)
    look(40, 55)
    return out


@pytest.mark.parametrize("integer", [False, True])
@pytest.mark.parametrize("n,max_delay", [(1100, 1), (2500, 3), (2500, 4), (2500, 16), (40_001, 9)])
def test_rows_between_launches(n, max_delay, integer):
    want = drive(S.SN_PULL_PLAIN, n, max_delay, integer)
    assert sum(int(S.unpack_raster(w, n).sum()) for w in want[9:10]) > 100
    for k, (a, b) in enumerate(zip(drive(0, n, max_delay, integer), want)):
        assert np.array_equal(a, b), k


def test_captured_run_after_a_reset():
    """A captured run of 20 steps from step 0, launched again after a reset and other
    runs, gives the same steps."""
    wl = W.random_small(64, n=2500, integer=True, steps=20, p=0.005, max_delay=16, events_rate=40.0)
    stream = torch.cuda.Stream()
    ctx = S.from_workload(wl, flags=S.SN_PROP_PULL, record_steps=20, stream=stream.cuda_stream)
    S.sn_run(ctx, 20)
    S.sn_sync(ctx)
    want = S.sn_get_spikes(ctx, 0, 20).copy()
    v = np.asarray(S.sn_get_state(ctx)[0]).copy()
    assert S.unpack_raster(want, 2500).sum() > 100
    S.sn_reset(ctx)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        S.sn_run(ctx, 20)
    for runs in ((), (1, 1, 1), (20,)):
        S.sn_reset(ctx)
        for q in runs:
            S.sn_run(ctx, q)
        S.sn_reset(ctx)
        with torch.cuda.stream(stream):
            graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(np.asarray(S.sn_get_state(ctx)[0]), v)


@pytest.mark.parametrize("max_delay,blocked", [(1, True), (3, False), (12, True)])
def test_form_of_wide_blocks(max_delay, blocked):
    """More than 672 neurons a block: with delays up to 3 the blocked kernel is the
    slower one (6.7 against 6.3 us a step) and the one-step kernel's store is built."""
    n, k = 140_000, 30
    rng = np.random.default_rng(max_delay)
    pre = np.repeat(np.arange(n, dtype=np.int32), k)
    args = (np.ones(n), np.zeros(n), np.zeros(n), np.zeros(n, np.int32), pre,
            rng.integers(0, n, n * k).astype(np.int32), np.full(n * k, 0.1, np.float32),
            rng.integers(1, max_delay + 1, n * k).astype(np.int32))
    auto, plain = (S.sn_pull_store_info(S.sn_create(*args, dtype="f32", max_delay=max_delay,
                                                    flags=S.SN_PROP_PULL | form)) for form in FORMS[:2])
    assert (auto != plain) == blocked

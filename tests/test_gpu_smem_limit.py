"""Host threads, each with a context of its own, launching the same kernel with
different amounts of shared memory: none may lower the process-wide limit under
another's launch.  All contexts run on one stream, so the kernels themselves run one
after another; only the host calls interleave."""

import threading

import numpy as np
import pytest

from paper_2305_02510_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CALLS = 8000


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()


def contexts(kind, stream):
    """Small networks and a large one of the same kernel instantiation."""
    from paper_2305_02510_gb300 import sn as S
    if kind == "dense":
        return [S.from_workload(W.large_dense(n=n, steps=1), flags=S.SN_DENSE_SLAB(1), record_steps=1, stream=stream)
                for n in (300, 300, 300, 2500)]
    form = {"pull": 0, "pull-plain": S.SN_PULL_PLAIN, "pull-coded": S.SN_PULL_CODED}[kind]
    return [S.from_workload(W.random_small(n, n=n, integer=False, steps=1, p=4.0 / n, max_delay=9),
                            flags=S.SN_PROP_PULL | form, record_steps=1, stream=stream)
            for n in (1100, 1100, 1100, 9000)]


@pytest.mark.parametrize("kind", ["pull", "pull-plain", "pull-coded", "dense"])
def test_launches_from_several_threads(kind):
    from paper_2305_02510_gb300 import sn as S
    stream = torch.cuda.Stream()
    ctxs = contexts(kind, stream.cuda_stream)
    errors = []

    def work(ctx):
        try:
            for k in range(CALLS):
                S.sn_run(ctx, 1)
                if k % 100 == 99:
                    S.sn_sync(ctx)
        except S.SnError as e:
            errors.append(str(e))

    threads = [threading.Thread(target=work, args=(c,)) for c in ctxs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert [S.sn_get_counters(c)[0] for c in ctxs] == [CALLS] * len(ctxs)

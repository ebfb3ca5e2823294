"""The shared dense network with one tile per block (spikes as tagged bits,
expanded into tensor memory): exact at the smallest and odd numbers of K blocks,
over runs that end anywhere in the operand ring, against the oracle per train;
and its overflow check."""

import numpy as np
import pytest

from oracle import compare
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


@pytest.mark.parametrize("n,trains", [(128, 128), (256, 384), (640, 128), (1152, 256)])
def test_runs(n, trains):
    runs = [1, 2, 3, 5, 14]
    T = sum(runs)
    wl = W.shared_dense_i8(n=n, batch=trains, steps=T)
    ctx = S.from_shared_workload(wl, record_steps=T)
    for q in runs:
        S.sn_run(ctx, q)
    bits = S.sn_get_spikes(ctx, 0, T)
    v, r = S.sn_get_state(ctx)
    w, total = n // 32, 0
    for b in (0, 31, 32, trains - 1):
        got = S.unpack_raster(np.ascontiguousarray(bits[:, b * w:(b + 1) * w]), n)
        compare.check_int_run(wl, got, v.reshape(trains, n)[b], r.reshape(trains, n)[b], T, net_index=b)
        total += int(got.sum())
    assert total > 0


@pytest.mark.parametrize("steps,overflows", [(255, False), (260, True)])
def test_overflow(steps, overflows):
    """2^23 a step into a neuron that never fires: 255 steps stay in int32."""
    n = 128
    ctx = S.sn_create_shared_dense_i8(np.full(n, np.inf), np.zeros(n), np.zeros(n), np.zeros(n, np.int32),
                                      np.zeros((n, n), np.int8), 128, record_steps=1)
    S.sn_set_poisson(ctx, np.arange(n), 1.0, 2.0 ** 23, 1)
    S.sn_run(ctx, steps)
    if overflows:
        with pytest.raises(S.SnError) as e:
            S.sn_sync(ctx)
        assert e.value.status == S.SN_EOVERFLOW
    else:
        S.sn_sync(ctx)
        v, _ = S.sn_get_state(ctx)
        assert int(v.max()) <= steps * 2 ** 23 and int(v.max()) >= (steps - 2) * 2 ** 23

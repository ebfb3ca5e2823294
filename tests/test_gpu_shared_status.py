"""A status latched by one block while others are at work ends a shared network's run
with that status, and the context's memory and later contexts stay usable: the waits
of every warp give up together.  One neuron of one tile leaves int32 (2^23 a step
into a neuron that never fires), its block latches that when it is done with the last
step, and the other tiles' blocks are then in theirs.  In the form with more tiles
than blocks the grid barriers are in between."""

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


@pytest.mark.parametrize("n,trains", [(2432, 1024), (2560, 1024)])   # 152 and 160 tiles
def test_overflow_of_one_tile(n, trains):
    for repeat in range(5):
        ctx = S.sn_create_shared_dense_i8(np.full(n, np.inf), np.zeros(n), np.zeros(n), np.zeros(n, np.int32),
                                          np.zeros((n, n), np.int8), trains, record_steps=1)
        S.sn_set_poisson(ctx, np.array([n - 1 - repeat]), 1.0, 2.0 ** 23, 1)
        S.sn_run(ctx, 260)
        with pytest.raises(S.SnError) as e:
            S.sn_sync(ctx)
        assert e.value.status == S.SN_EOVERFLOW
        del ctx
    ctx = S.sn_create_shared_dense_i8(np.full(n, np.inf), np.zeros(n), np.zeros(n), np.zeros(n, np.int32),
                                      np.zeros((n, n), np.int8), trains, record_steps=1)
    S.sn_set_poisson(ctx, np.array([7]), 1.0, 2.0 ** 23, 1)
    S.sn_run(ctx, 200)
    S.sn_sync(ctx)
    v, _ = S.sn_get_state(ctx)
    assert int(v.max()) >= 198 * 2 ** 23 and np.count_nonzero(v) == trains

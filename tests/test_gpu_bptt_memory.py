"""A feedforward context short of memory: the k-th device allocation of its creation
fails (host-side injection, SN_FAULT_ALLOC_AT).  One buffer of spikes per layer is a
convenience: where one of them cannot be had, a single buffer serves all layers and
the tensor cores stay in use, with the same bits.  Only the weight parts, the
gradient operand and that single buffer are needed, and a context that does without
the tensor cores holds none of their buffers."""

import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES, BATCH, STEPS = (70, 200, 130, 20), 64, 60


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()


def test_tensor_cores_without_a_spike_buffer_per_layer():
    from paper_2305_02510_gb300 import bptt, sn as S
    layers = len(SIZES) - 1
    rng = np.random.default_rng(5)
    x = torch.from_numpy((rng.random((STEPS, BATCH, SIZES[0])) < 0.2).astype(np.uint8)).cuda()
    ws = [torch.from_numpy(rng.normal(0, np.sqrt(2.0 / a), (a, b)).astype(np.float32)).cuda().requires_grad_()
          for a, b in zip(SIZES[:-1], SIZES[1:])]
    ds = [rng.integers(1, 5, (a, b)).astype(np.uint8) for a, b in zip(SIZES[:-1], SIZES[1:])]
    gc = torch.from_numpy(rng.normal(0, 1, (BATCH, SIZES[-1])).astype(np.float32)).cuda()

    def step(net):
        counts = bptt.SNNFunction.apply(net, x, *ws)
        return [counts.detach(), *torch.autograd.grad(counts, ws, gc)]

    def held():
        free = torch.cuda.mem_get_info()[0]
        net = bptt.FFNet(SIZES, ds, batch=BATCH, steps=STEPS)
        return net, free - torch.cuda.mem_get_info()[0]

    net, full = held()
    want = step(net)
    del net
    tensor = []
    try:
        for k in range(1, 200):
            os.environ["SN_FAULT_ALLOC_AT"] = str(k)
            try:
                net, held_bytes = held()
            except S.SnError:
                continue
            finally:
                os.environ.pop("SN_FAULT_ALLOC_AT")
            try:
                S.sn_ff_set_engine(net.ctx, S.SN_FF_TENSOR)
                tensor.append(True)
                for a, b in zip(step(net), want):
                    assert torch.equal(a, b), k
            except S.SnError as e:
                assert e.status == S.SN_EUNSUPPORTED
                tensor.append(False)
                assert held_bytes < full, k
            del net
            if len(tensor) > 3 * layers + 3:
                break
    finally:
        os.environ.pop("SN_FAULT_ALLOC_AT", None)
    # two weight operands a layer and the gradient, then the layers' spikes
    assert tensor == [False] * (2 * layers + 1) + [True] * (layers + 3), tensor

"""New memory at the address of a prepared workspace is not taken for the prepared one: the
split of W_r that dmoe_router_prepare wrote is gone, and the next forward writes it again."""
import pytest
import torch

from dmoe_synth import TINY
from tests import parity as P

pytestmark = pytest.mark.gpu


def test_initialised_workspace_is_not_prepared():
    shape = TINY.with_(block_size=32, n_blocks=4, n_experts=32)   # the tensor-core router
    m = P.dm()
    dev, _ = P.make(shape, seed=3)
    from paper_2605_30876_gb300.layer import MoELayer
    layer = MoELayer.from_shape(shape, dev)   # prepares its workspace
    y = layer.forward(dev["x"]).clone()
    probs = torch.empty((shape.T, shape.n_experts), device="cuda")

    def scores(ws):
        out = torch.empty_like(probs)
        m.dmoe_router(layer.desc, dev["x"], dev["w_r"], dev["bias"], layer.topk_idx,
                      layer.topk_gate, None, None, out, workspace=ws)
        return out

    want = scores(layer.ws)
    m.dmoe_workspace_init(layer.ws)           # as new memory at the same address would be
    assert torch.equal(scores(layer.ws), want)
    m.dmoe_router_prepare(layer.desc, dev["w_r"], layer.ws)
    addr = layer.ws.data_ptr()
    layer.ws = None                           # torch's allocator hands the block out again
    ws = m.alloc_workspace(layer.desc)
    assert ws.data_ptr() == addr
    assert torch.equal(scores(ws), want)
    layer.ws = ws
    assert torch.equal(layer.forward(dev["x"]), y)

"""The record of a prepared workspace (the split of W_r that dmoe_router_prepare wrote). New memory at
the address of a prepared workspace is not taken for the prepared one: the split is gone, and the
next forward writes it again. Calls with another layout neither take the split for theirs nor leave
it marked as valid once they have written over it."""
import pytest
import torch

from dmoe_synth import ROUTE_TOKEN, TINY
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


# a workspace prepared for 64 blocks of 32 tokens, then used for calls whose layouts differ: the
# split elsewhere by a few hundred bytes (token routing has no coreset words before it), at half
# the size, and a router that has no split and more scratch than the first layout before it
OTHERS = {
    "token": dict(mode=ROUTE_TOKEN),
    "fewer_blocks": dict(n_blocks=32),
    "no_split": dict(n_experts=24, d_ff=512),
}


@pytest.mark.parametrize("name", OTHERS)
def test_a_workspace_shared_by_two_layouts(name):
    base = TINY.with_(block_size=32, n_blocks=64, n_experts=32, top_k=8)
    other = base.with_(**OTHERS[name])
    m = P.dm()
    dev, _ = P.make(base, seed=5)
    dev2, _ = P.make(other, seed=5)
    if other.n_experts == base.n_experts:    # the same router weight: only the layouts differ
        dev2["w_r"], dev2["bias"] = dev["w_r"], dev["bias"]
    want, want2 = P.gpu_router(base, dev), P.gpu_router(other, dev2)   # workspaces of their own
    size = max(m.dmoe_workspace_size(P.desc_of(s)) for s in (base, other))
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    m.dmoe_workspace_init(ws)
    m.dmoe_router_prepare(P.desc_of(base), dev["w_r"], ws)

    def check(shape, d, w):
        got = P.gpu_router(shape, d, ws=ws)
        for key in w:
            assert (got[key] == w[key]).all(), key

    def forward(shape, d, w):
        desc = P.desc_of(shape)
        if w is None:
            w = m.alloc_workspace(desc)
        y = torch.empty((shape.T, shape.d_model), dtype=torch.bfloat16, device="cuda")
        m.dmoe_layer_forward(desc, d["x"], d["w_r"], d["bias"], d["w_gate"], d["w_up"], d["w_down"],
                             None, None, None, y, workspace=w)
        assert m.dmoe_get_device_error(w)[0] == 0
        return y

    check(base, dev, want)
    check(other, dev2, want2)
    check(base, dev, want)
    m.dmoe_router_prepare(P.desc_of(base), dev["w_r"], ws)
    assert torch.equal(forward(other, dev2, ws), forward(other, dev2, None))
    check(base, dev, want)
    assert torch.equal(forward(base, dev, ws), forward(base, dev, None))

"""The expert launches where their tiles can go wrong, against the CPU oracle. The general one (more
than 64 tokens): tiles of 32 to 256 token rows with remainders, blocks that fill half tiles in twos or
fours, blocks that fill none, d and I of an odd number of 128-row tiles, more token tiles than
one, and fewer units than clusters. The decode-size one: both unit heights, the smallest and the
largest token count, and outputs kept by few tokens. Both with every form of the gate and up
weights' copies: one copy for both tensors, the gate's or the up's address the lower one, in the
routed experts and the shared one apart; and a copy for each, which any pair that is one tensor
(distance 0 is no stride) brings about for the other pair too."""
import numpy as np
import pytest
import torch

import oracle as O
from dmoe_synth import ROUTE_TOKEN, TINY
from tests import parity as P

pytestmark = pytest.mark.gpu

SMALL = TINY.with_(n_experts=32, top_k=4, d_ff_shared=128, bias_scale=0.5)
CASES = {
    # block top-k read block by block: half tiles of whole blocks (a multiple of 2 or 4 blocks)
    "blocks_24x5": SMALL.with_(block_size=24, n_blocks=5),
    "blocks_40x4_d384": SMALL.with_(block_size=40, n_blocks=4, d_model=384),
    "blocks_8x33": SMALL.with_(block_size=8, n_blocks=33, n_experts=8),
    "blocks_128x3": SMALL.with_(block_size=128, n_blocks=3),
    "blocks_256x3": SMALL.with_(block_size=256, n_blocks=3),   # two halves, a CTA's each
    "blocks_48x9_d640": SMALL.with_(block_size=48, n_blocks=9, d_model=640, n_experts=16),
    # no half tile of whole blocks: the copied rows
    "blocks_72x3": SMALL.with_(block_size=72, n_blocks=3),
    "blocks_33x8_p07": SMALL.with_(block_size=33, n_blocks=8, top_p=0.7),
    "blocks_32x10_p06_fewer": SMALL.with_(n_blocks=10, block_size=32, top_p=0.6, top_k=3,
                                          block_top_k=4),
    # token routing: the fewest tokens, remainders of 1 and 44 rows in a second token tile
    "token_65_k1": SMALL.with_(block_size=13, n_blocks=5, mode=ROUTE_TOKEN, top_k=1,
                               d_ff_shared=0),
    "token_257_all": SMALL.with_(block_size=257, n_blocks=1, mode=ROUTE_TOKEN, n_experts=8,
                                 top_k=8),
    "token_300_d384_I384": SMALL.with_(block_size=60, n_blocks=5, mode=ROUTE_TOKEN, n_experts=8,
                                       top_k=8, d_model=384, d_ff=384, d_ff_shared=256),
    # decode size: 32-row gate/up units (few experts) and 64-row ones, 1 to 64 tokens
    "decode_1": SMALL.with_(block_size=1, n_blocks=1),
    "decode_5x12": SMALL.with_(block_size=12, n_blocks=5),
    "decode_64_all": SMALL.with_(block_size=64, n_blocks=1, n_experts=8, top_k=8, d_model=512),
    "decode_token_61": SMALL.with_(block_size=61, n_blocks=1, mode=ROUTE_TOKEN, n_experts=256,
                                   top_k=16, d_ff=256, d_ff_shared=512),
    "decode_d384_p06": SMALL.with_(block_size=17, n_blocks=3, top_p=0.6, d_model=384),
}


# (routed, shared): 0: the up tensor is the gate tensor; 1: gate at the lower address; 2: up there
FORMS = {"gate_first": (1, 1), "up_first": (2, 2), "shared_up_first": (1, 2), "one_tensor": (0, 0),
         "routed_apart": (1, 0), "routed_apart_up_first": (2, 0), "shared_apart": (0, 1)}


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("name", CASES)
def test_layer_matches_oracle(name, form):
    shape = CASES[name]
    m = P.dm()
    dev, host = P.make(shape, seed=7)
    for prefix, how in zip(("w", "ws"), FORMS[form]):
        gate, up = f"{prefix}_gate", f"{prefix}_up"
        if dev[gate] is None:
            continue
        if how == 0:
            dev[up], host[up] = dev[gate], host[gate]
            continue
        both = torch.stack([dev[gate], dev[up]] if how == 1 else [dev[up], dev[gate]])
        dev[gate], dev[up] = both[how - 1], both[2 - how]
    from paper_2605_30876_gb300.layer import MoELayer
    layer = MoELayer.from_shape(shape, dev)
    y = layer.forward(dev["x"]).clone()
    st, info = m.dmoe_get_device_error(layer.ws)
    assert st == 0, info
    idx = layer.topk_idx.cpu().numpy()
    orc = P.oracle_routing(shape, host)
    assert int(layer.n_unique.item()) == len(np.unique(idx))
    P.check_output(y, P.oracle_output(host, idx, orc.scores), label=name)
    assert torch.equal(y, layer.forward(dev["x"]))
    # the same routing through the dispatch and the experts called on their own (gathered rows)
    gate = torch.from_numpy(O.gates_for(orc.scores, idx).astype(np.float32)).cuda()
    out, ws = P.gpu_dispatch(shape, layer.topk_idx)
    y2 = torch.empty_like(y)
    m.dmoe_moe_forward(layer.desc, dev["x"], dev["w_gate"], dev["w_up"], dev["w_down"],
                       dev["ws_gate"], dev["ws_up"], dev["ws_down"], gate, out["n_unique"],
                       out["unique_ids"], out["offsets"], out["rows"], out["pos"], y2, workspace=ws)
    st, info = m.dmoe_get_device_error(ws)
    assert st == 0, info
    P.check_output(y2, P.oracle_output(host, idx, orc.scores), label=name + " experts")

"""Experts on a dispatch that recorded a fault: the entries that it left unwritten in the caller's rows
and pos (here far out of range) are not followed, and the fault is what the next reading of the
workspace's record gives. Decode size and the general launches, both sizes of the dispatch."""
import numpy as np
import pytest
import torch

from dmoe_synth import ROUTE_TOKEN, TINY
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [33, 96, 545])
@pytest.mark.parametrize("fault", ["id", "twice"])
@pytest.mark.parametrize("poison", [2 ** 31 - 1, -2 ** 31])
def test_experts_after_a_bad_dispatch(T, fault, poison):
    k, E = 2, 16
    shape = TINY.with_(block_size=T, n_blocks=1, mode=ROUTE_TOKEN, n_experts=E, top_k=k)
    dev, _ = P.make(shape, seed=T)
    m, desc = P.dm(), P.desc_of(shape)
    ws = m.alloc_workspace(desc)

    def buf(n, v):
        return torch.full((n,), v, dtype=torch.int32, device="cuda")

    def forward(idx):
        out = [buf(1, poison), buf(E, poison), buf(E + 1, poison), buf(T * k, poison),
               buf(T * k, poison)]
        y = torch.empty((T, shape.d_model), dtype=torch.bfloat16, device="cuda")
        gate = torch.full((T, k), 0.5, device="cuda")
        m.dmoe_dispatch(desc, torch.from_numpy(idx).cuda(), *out, workspace=ws)
        m.dmoe_moe_forward(desc, dev["x"], dev["w_gate"], dev["w_up"], dev["w_down"], None, None,
                           None, gate, *out, y, workspace=ws)
        return y

    good = np.stack([np.arange(T) % E, (np.arange(T) + 1) % E], 1).astype(np.int32)
    want = forward(good)
    assert m.dmoe_get_device_error(ws)[0] == 0
    bad = good.copy()
    bad[T // 2, 1] = E if fault == "id" else bad[T // 2, 0]
    forward(bad)
    assert m.dmoe_get_device_error(ws)[0] == 5
    assert torch.equal(forward(good), want)      # the workspace is as before
    assert m.dmoe_get_device_error(ws)[0] == 0

"""Decode size, more than 48 tokens: a token's output has the same bits whichever height the gate/up
units take (32 or 64 rows, by the count of unique experts), so it does not depend on how the other
tokens are routed."""
import numpy as np
import pytest
import torch

from dmoe_synth import ROUTE_TOKEN, TINY
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [49, 64])
@pytest.mark.parametrize("d,I,Is", [(512, 256, 0), (2048, 512, 512)])
def test_output_is_the_same_with_few_and_with_many_experts(T, d, I, Is):
    E, k, kept = 128, 2, 16
    shape = TINY.with_(block_size=T, n_blocks=1, mode=ROUTE_TOKEN, n_experts=E, top_k=k, d_model=d,
                       d_ff=I, d_ff_shared=Is)
    dev, _ = P.make(shape, seed=T)
    m, desc = P.dm(), P.desc_of(shape)
    gate = torch.full((T, k), 0.5, device="cuda")

    def forward(idx):
        out, ws = P.gpu_dispatch(shape, torch.from_numpy(idx).cuda())
        y = torch.empty((T, d), dtype=torch.bfloat16, device="cuda")
        m.dmoe_moe_forward(desc, dev["x"], dev["w_gate"], dev["w_up"], dev["w_down"],
                           dev["ws_gate"], dev["ws_up"], dev["ws_down"], gate, out["n_unique"],
                           out["unique_ids"], out["offsets"], out["rows"], out["pos"], y,
                           workspace=ws)
        assert m.dmoe_get_device_error(ws)[0] == 0
        return y[:kept], int(out["n_unique"].item())

    few = np.tile(np.array([3, 70], np.int32), (T, 1))
    many = few.copy()
    many[kept:] = np.arange(2 * (T - kept)).reshape(-1, 2)
    (a, ua), (b, ub) = forward(few), forward(many)
    # units of 32 rows where all of them fit one round of 152 CTAs, else of 64
    assert (ua * I + Is) // 32 <= 152 < (ub * I + Is) // 32
    assert torch.equal(a, b)

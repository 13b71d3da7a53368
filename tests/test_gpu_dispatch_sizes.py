"""dmoe_dispatch against the oracle around the size where it becomes one launch (512 tokens), at
chunk remainders, the smallest and the largest k and E, and its fault record on both sides."""
import numpy as np
import pytest
import torch

from dmoe_synth import ROUTE_TOKEN, TINY
from tests import parity as P

pytestmark = pytest.mark.gpu

# tokens, experts, k
SIZES = [(1, 8, 1), (33, 16, 16), (64, 256, 8), (511, 256, 16), (512, 8, 8), (513, 8, 8),
         (545, 256, 16), (1024, 64, 3), (4096, 256, 16)]


def shape_of(T, E, k):
    return TINY.with_(block_size=T, n_blocks=1, mode=ROUTE_TOKEN, n_experts=E, top_k=k)


@pytest.mark.parametrize("T,E,k", SIZES)
def test_dispatch_matches_oracle(T, E, k):
    shape = shape_of(T, E, k)
    rng = np.random.default_rng(T * 7 + E + k)
    pop = rng.random(E) ** 3 + 1e-3     # skewed: some experts with no token at small T
    idx = np.stack([rng.choice(E, k, replace=False, p=pop / pop.sum()) for _ in range(T)])
    idx = idx.astype(np.int32)
    idx_t = torch.from_numpy(idx).cuda()
    out, ws = P.gpu_dispatch(shape, idx_t)
    assert P.dm().dmoe_get_device_error(ws)[0] == 0
    P.check_dispatch(shape, idx, out)


@pytest.mark.parametrize("T", [512, 513])
@pytest.mark.parametrize("fault,code", [("id", 2), ("twice", 3)])
def test_dispatch_records_bad_ids(T, fault, code):
    shape = shape_of(T, 16, 2)
    idx = np.stack([np.arange(T) % 16, (np.arange(T) + 1) % 16], 1).astype(np.int32)
    idx[T - 1, 1] = 16 if fault == "id" else idx[T - 1, 0]
    _, ws = P.gpu_dispatch(shape, torch.from_numpy(idx).cuda())
    st, info = P.dm().dmoe_get_device_error(ws)
    # 4 (the pairs do not add up) can be recorded first only where the one launch both counts and
    # checks, and only for the bad id: a doubled expert's pairs are all counted there
    assert st == 5 and info[0] in ((code, 4) if T == 512 and fault == "id" else (code,))

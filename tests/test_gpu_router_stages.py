"""The tensor-core router's scores and selection at each number of stages its slices take: one
stage per chunk of 64 of d where shared memory holds them, fewer with many experts in a CTA."""
import pytest

from dmoe_synth import ROUTE_TOKEN, TINY
from tests import parity as P

pytestmark = pytest.mark.gpu

# tokens, d, experts            experts per CTA, chunks, stages
SIZES = [(128, 128, 32),      # 32, 1, 2 (the fewest)
         (2048, 384, 256),    # 64, 3, 3
         (256, 2048, 128),    # 32, 4, 4
         (1025, 1024, 256),   # 64, 4, 4; the last tile has one row
         (2048, 2048, 128),   # 128, 4, 3: the first stage is taken twice
         (4096, 1280, 160),   # 160, 4, 2: each stage is taken twice
         (4096, 1280, 256)]   # 256, 4, 2


@pytest.mark.parametrize("T,d,E", SIZES)
def test_router_matches_oracle(T, d, E):
    shape = TINY.with_(block_size=T, n_blocks=1, mode=ROUTE_TOKEN, n_experts=E, top_k=8,
                       d_model=d)
    dev, host = P.make(shape, seed=T + d + E)
    P.check_routing(shape, P.gpu_router(shape, dev), P.oracle_routing(shape, host))

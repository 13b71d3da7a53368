"""Algorithm 1 by counting, against the oracle. 0 < p < 1: the sorted prefix at the counts of
nonzero experts where the work is split another way (8, 4, 2 or 1 threads an expert, pairs with an
odd end). Block top-k: the smallest and largest k, partly filled warps, equal sums."""
import numpy as np
import pytest
import torch

from dmoe_synth import ROUTE_BLOCK, TINY, to_numpy
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [0.1, 0.9])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256])
def test_coreset_is_the_oracles_prefix(n, p):
    # 256 tokens, token t's best expert is (37 t) mod n: exactly n experts are kept once
    B = d = E = 256
    shape = TINY.with_(block_size=B, n_blocks=1, mode=ROUTE_BLOCK, n_experts=E, top_k=1,
                       top_p=p, d_model=d)
    rng = np.random.default_rng(n)
    w_r = np.zeros((d, E), np.float32)
    w_r[np.arange(B), 37 * np.arange(B) % n] = rng.uniform(2, 8, B)
    dev = dict(x=torch.eye(B, d).bfloat16().cuda(), w_r=torch.from_numpy(w_r).cuda(),
               bias=torch.zeros(E).cuda())
    orc = P.oracle_routing(shape, to_numpy(dev))
    g = P.gpu_router(shape, dev)
    P.check_routing(shape, g, orc)
    # descending sums, up to the scores' tolerance (1e-5 relative, summed over the block)
    S = np.zeros(E)
    for t in range(B):
        S[37 * t % n] += orc.scores[t, 37 * t % n]
    v = S[g["coreset"][0][:int(g["coreset_size"][0])]]
    assert np.all(v[:-1] >= v[1:] - 1e-5 * v.max())


@pytest.mark.parametrize("nb", [1, 3])       # the decode-size launch and the general one
@pytest.mark.parametrize("E,k", [(8, 1), (8, 8), (40, 9), (256, 1), (256, 8), (256, 9), (256, 16)])
def test_block_top_k_coreset(E, k, nb):
    shape = TINY.with_(block_size=32, n_blocks=nb, mode=ROUTE_BLOCK, n_experts=E, top_k=k,
                       top_p=0.0, d_model=256)
    dev, host = P.make(shape, seed=E + k)
    g = P.gpu_router(shape, dev)
    P.check_routing(shape, g, P.oracle_routing(shape, host))
    # every score equal: every token keeps the k lowest ids, and so does the block, in order
    dev["w_r"].zero_()
    dev["bias"].zero_()
    g = P.gpu_router(shape, dev)
    assert np.array_equal(g["coreset"][:, :k], np.tile(np.arange(k), (nb, 1)))
    assert np.all(g["coreset_size"] == k) and np.array_equal(g["idx"], np.tile(np.arange(k), (32 * nb, 1)))

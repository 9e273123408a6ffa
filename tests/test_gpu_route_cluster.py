"""Prefill routing on clusters (many experts, long rows; route_tile_cluster_kernel) against the oracle:
token counts at the edges of the 64- and 128-token tiles, expert counts that fill no whole column tile,
contractions whose eighth is uneven or no multiple of a stage, every routing mode."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_34077_gb300 import inputs as I
from paper_2609_34077_gb300 import mcft as M
from tests.gpu_helpers import check_routing, f64

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("d,E,K,T", [(1024, 17, 2, 65), (1088, 33, 8, 127), (2048, 64, 6, 129),
                                     (1984, 25, 5, 64 * 3), (1024, 64, 1, 2048), (1152, 40, 4, 2049),
                                     (4096, 63, 7, 2100)])
@pytest.mark.parametrize("mode", [M.MCFT_ROUTE_TOPK, M.MCFT_ROUTE_HARD_MASK, M.MCFT_ROUTE_SOFT_PRIOR])
def test_route_clusters(d, E, K, T, mode):
    shape = I.LayerShape(f"route-{d}-{E}", d=d, E=E, K=K, w=64, n_shared=0, gate=(T + K) % 2,
                         dtype=I.BF16, cache_slots=2, keep=max(K, E // 2))
    x, w = I.hidden_iid(400 + T, shape, T), I.router_weight(400 + E, shape)
    mask = I.keep_mask(400, E, shape.keep)
    extra = {M.MCFT_ROUTE_TOPK: {}, M.MCFT_ROUTE_HARD_MASK: dict(mask=mask),
             M.MCFT_ROUTE_SOFT_PRIOR: dict(prior=I.prior_from_mask(mask))}[mode]
    idx, gate = M.mcft_route(M.desc_of(shape), x.to(DEV), w.to(DEV), mode, **extra)
    M.mcft_device_error()
    ref = oracle.routing.route(f64(x), f64(w), K, mode, shape.gate, **extra)
    flagged, _ = check_routing(idx, gate, ref, shape.gate)
    assert flagged <= T // 10


@pytest.mark.parametrize("d,E,K,T", [(64, 5, 3, 1), (2048, 64, 6, 9), (2048, 64, 6, 70), (256, 16, 4, 70)])
def test_ties_and_infinities(d, E, K, T):
    """Equal scores go to the lower index (zeros of either sign are equal), and -inf scores rank last
    but stay eligible."""
    desc = M.LayerDesc(d, E, K, 64, 0, I.GATE_PLAIN, M.MCFT_BF16)
    x = torch.zeros(T, d, dtype=torch.bfloat16, device=DEV)
    x[:, 0] = 1.0
    w = torch.zeros(E, d, dtype=torch.bfloat16, device=DEV)
    w[0, 0] = -0.0
    w[E - 1, 0] = 1.0
    w[1, 0] = float("-inf")
    idx, _ = M.mcft_route(desc, x, w, M.MCFT_ROUTE_TOPK)
    # every product with the other (zero) elements is 0, so expert 1 has a NaN-free -inf only if x is 0
    # nowhere else; its score is -inf + 0 = -inf
    M.mcft_device_error()
    want = ([E - 1, 0] + list(range(2, E - 1)) + [1])[:K]
    assert np.array_equal(idx.cpu().numpy(), np.tile(np.array(want, np.int32), (T, 1)))

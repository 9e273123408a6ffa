"""Decode work items that grow with the number of items (csrc/ffn_decode.cu, widen_item): a layer just
large enough for 64-row GEMM13 items, against the oracle, and the same bits from the plain forward, the
cached forward (hits and fetched misses, in one launch up to 16 tokens and in two above), and the
forward with adapters that add nothing (the separate GEMM13 kernel)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_34077_gb300 import inputs as I
from paper_2609_34077_gb300 import mcft as M
from tests.gpu_helpers import TOL_BF16, check_output, expert_triples, f64, shared_triples, weights

pytestmark = pytest.mark.gpu
DEV = "cuda"
# 65 segments x 1088 / 64 rows = 1105 items, over 3.5 rounds of 304; 1024 wide would stay at 32 rows
SHAPE = I.LayerShape("wide-items", d=2048, E=64, K=6, w=1088, n_shared=1, gate=I.GATE_RENORM,
                     dtype=I.BF16, cache_slots=20, keep=64)


@pytest.mark.parametrize("T", [11, 40])
def test_wide_items(T):
    lw = weights(SHAPE, 500)
    desc = M.desc_of(SHAPE)
    x = I.ar1_streams(500, SHAPE, 1, T)[0]
    ids = I.random_ids(501, 1, T, SHAPE.K, SHAPE.E)[0]
    gate = np.random.default_rng(502).uniform(0.05, 1.0, ids.shape).astype(np.float32)
    host = [b.pin_memory() for b in lw.experts]
    experts = [b.to(DEV) for b in lw.experts]
    shared = [b.to(DEV) for b in lw.shared]
    xd, idx, g = x.to(DEV), torch.from_numpy(ids).to(DEV), torch.from_numpy(gate).to(DEV)
    y = M.mcft_moe_forward(desc, xd, idx, g, experts, shared)
    M.mcft_device_error()
    ref = oracle.ffn.moe_layer(f64(x), ids, gate.astype(np.float64), expert_triples(lw, SHAPE),
                               shared_triples(lw, SHAPE))
    check_output(y, ref, TOL_BF16, f"T={T}")
    cache = M.mcft_cache_create(1, SHAPE.E, SHAPE.cache_slots, SHAPE.expert_bytes, host,
                                max_assign=T * SHAPE.K)
    copy = torch.cuda.Stream()
    for _ in range(2):  # first fills and bypasses, then hits beside misses
        M.mcft_cache_step(cache, 0, idx)
        yc = M.mcft_moe_forward_cached(desc, xd, idx, g, cache, 0, shared, copy_stream=copy)
        torch.cuda.synchronize()
        assert torch.equal(yc, y)
    yl = M.mcft_moe_forward_lora(desc, xd, idx, g, experts, shared, [None] * 64, [None], 8, 2.0)
    M.mcft_device_error()
    assert torch.equal(yl, y)

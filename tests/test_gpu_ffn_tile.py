"""The fp32 FFN in 64-token tiles (csrc/ffn_tile.cu) against the oracle: segments at the edges of the
16-token warps and 64-token tiles, one and several contraction steps, adapters, and the cached forward,
which computes the hits and the fetched experts in two launches and must give the plain forward's bits."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_34077_gb300 import inputs as I
from paper_2609_34077_gb300 import mcft as M
from tests.gpu_helpers import TOL_F32, check_output, expert_triples, f64, shared_triples, weights
from tests.test_gpu_rows import _sized_ids

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _shape(d, w, E=4, S=0):
    return I.LayerShape(f"tile-{d}x{w}-S{S}", d=d, E=E, K=2, w=w, n_shared=S, gate=I.GATE_RENORM,
                        dtype=I.F32, cache_slots=2, keep=E)


def _args(shape, T, ids, seed):
    lw = weights(shape, seed)
    x = I.hidden_iid(seed + 1, shape, T)
    gate = np.random.default_rng(seed).uniform(0.05, 1.0, ids.shape).astype(np.float32)
    dev = (M.desc_of(shape), x.to(DEV), torch.from_numpy(ids).to(DEV), torch.from_numpy(gate).to(DEV),
           [b.to(DEV) for b in lw.experts], [b.to(DEV) for b in lw.shared])
    ref = (f64(x), ids, gate.astype(np.float64), expert_triples(lw, shape), shared_triples(lw, shape))
    return dev, ref


@pytest.mark.parametrize("d,w,S", [(64, 64, 0), (128, 192, 1), (256, 512, 0)])
@pytest.mark.parametrize("T,first", [(24, [1, 16]), (70, [17, 64]), (130, [65, 127]), (300, [129])])
def test_tiles_against_the_oracle(d, w, S, T, first):
    shape = _shape(d, w, S=S)
    dev, ref = _args(shape, T, _sized_ids(T, 2, 4, first), 300 + T)
    y = M.mcft_moe_forward(*dev)
    M.mcft_device_error()
    check_output(y, oracle.ffn.moe_layer(*ref), TOL_F32, shape.name)


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3e38])
@pytest.mark.parametrize("k", [0, 40, 255])
def test_infinities_as_on_the_row_path(value, k):
    """An infinite, undefined or overflowing input in any step of the contraction: the token's outputs are
    infinite and undefined where the row-wise kernels' (a batch of one token) are; other tokens finite."""
    shape, T = _shape(256, 128), 70
    ids = _sized_ids(T, 2, 4, [17, 64])
    dev, _ = _args(shape, T, ids, 330)
    dev[1][3, k] = value
    y = M.mcft_moe_forward(*dev)
    y1 = M.mcft_moe_forward(dev[0], *(v[3:4].contiguous() for v in dev[1:4]), *dev[4:])
    M.mcft_device_error()
    assert torch.equal(torch.isnan(y[3:4]), torch.isnan(y1)) and torch.equal(torch.isinf(y[3:4]), torch.isinf(y1))
    assert torch.isfinite(torch.cat([y[:3], y[4:]])).all()


@pytest.mark.parametrize("rank", [8, 16])
def test_tiles_with_adapters(rank):
    shape, T, seed = _shape(128, 192, S=1), 90, 310
    dev, ref = _args(shape, T, _sized_ids(T, 2, 4, [65, 17]), seed)
    ad = [I.lora_block(seed, shape, e, rank) if e != 1 else None for e in range(4)]
    sad = [I.lora_block(seed, shape, ("shared", 0), rank)]
    put = lambda bs: [None if b is None else b.to(DEV) for b in bs]
    y = M.mcft_moe_forward_lora(*dev, put(ad), put(sad), rank, 16.0 / rank)
    M.mcft_device_error()
    split = lambda b: None if b is None else tuple(f64(t) for t in I.split_lora(b, shape, rank))
    check_output(y, oracle.ffn.moe_layer(*ref, lora=[split(b) for b in ad], shared_lora=[split(sad[0])],
                                         lora_scale=16.0 / rank), TOL_F32, "adapters")
    for b in ad + sad:  # up matrices of zero: the plain forward's bits
        for i, t in enumerate(I.split_lora(b, shape, rank) if b is not None else ()):
            if i % 2 == 1:
                t.zero_()
    y0 = M.mcft_moe_forward_lora(*dev, put(ad), put(sad), rank, 2.0)
    assert torch.equal(y0, M.mcft_moe_forward(*dev))


def test_cached_forward_gives_the_plain_bits():
    shape, T, seed = _shape(128, 192, S=1), 70, 320
    host = [b.pin_memory() for b in weights(shape, seed).experts]
    cache = M.mcft_cache_create(1, 4, 2, shape.expert_bytes, host, max_assign=2 * T)
    for ids in (_sized_ids(T, 2, 4, [17, 64]), _sized_ids(T, 2, 4, [64])):  # first fills, then hits too
        dev, _ = _args(shape, T, ids, seed)
        M.mcft_cache_step(cache, 0, dev[2])
        yc = M.mcft_moe_forward_cached(*dev[:4], cache, 0, dev[5], copy_stream=torch.cuda.Stream())
        torch.cuda.synchronize()
        M.mcft_device_error()
        assert torch.equal(yc, M.mcft_moe_forward(*dev))

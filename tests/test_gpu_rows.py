"""The expert GEMMs with the weight rows on the MMA's M side (csrc/gemm_rows.cu): layers whose hidden
size and width are any multiple of 64, and expert segments of any number of rows, against the oracle
(Section 3.1's gated sum of SwiGLU experts). Segment sizes sit at the edges of the token tiles (32 and
256 rows), sizes at the edges of the weight tiles (64, 128 and 256 rows)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_34077_gb300 import inputs as I
from paper_2609_34077_gb300 import mcft as M
from tests.gpu_helpers import TOL_BF16, check_output, expert_triples, f64, shared_triples, weights

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _shape(d, w, E=8, K=2, S=0):
    return I.LayerShape(f"rows-{d}x{w}-E{E}-S{S}", d=d, E=E, K=K, w=w, n_shared=S, gate=I.GATE_RENORM,
                        dtype=I.BF16, cache_slots=max(2, E // 2), keep=E)


def _sized_ids(T, K, E, first):
    """ids [T, K]: expert 0 gets exactly first[0] tokens, expert 1 first[1], ...; the others share
    the rest (K distinct ids per token)."""
    ids = np.empty((T, K), np.int32)
    left = list(first)
    for t in range(T):
        row = [e for e in range(len(left)) if left[e] > 0][:K]
        for e in row:
            left[e] -= 1
        n = len(first)
        row += [n + (t + j) % (E - n) for j in range(K - len(row))]
        ids[t] = row
    assert not any(left)
    return ids


def _run(shape, T, ids, seed, rank=0):
    lw = weights(shape, seed)
    desc = M.desc_of(shape)
    x = I.hidden_iid(seed + 1, shape, T)
    gate = np.random.default_rng(seed).uniform(0.05, 1.0, ids.shape).astype(np.float32)
    args = (desc, x.to(DEV), torch.from_numpy(ids).to(DEV), torch.from_numpy(gate).to(DEV),
            [b.to(DEV) for b in lw.experts], [b.to(DEV) for b in lw.shared])
    lora = dict()
    if rank:
        ad = [I.lora_block(seed, shape, e, rank) if e % 3 != 1 else None for e in range(shape.E)]
        sad = [I.lora_block(seed, shape, ("shared", s), rank) for s in range(shape.n_shared)]
        y = M.mcft_moe_forward_lora(*args, [None if b is None else b.to(DEV) for b in ad],
                                    [b.to(DEV) for b in sad], rank, 16.0 / rank)
        split = lambda b: None if b is None else tuple(f64(t) for t in I.split_lora(b, shape, rank))
        lora = dict(lora=[split(b) for b in ad], shared_lora=[split(b) for b in sad],
                    lora_scale=16.0 / rank)
    else:
        y = M.mcft_moe_forward(*args)
    M.mcft_device_error()
    ref = oracle.ffn.moe_layer(f64(x), ids, gate.astype(np.float64), expert_triples(lw, shape),
                               shared_triples(lw, shape), **lora)
    check_output(y, ref, TOL_BF16, f"{shape.name} T={T} rank={rank}")
    return args, y


@pytest.mark.parametrize("d,w", [(64, 64), (128, 192), (320, 64), (256, 128), (960, 704)])
@pytest.mark.parametrize("T,first", [(65, [1, 31]), (260, [32, 33]), (600, [255, 256, 257]),
                                     (700, [513, 64])])
def test_sizes_and_segments(d, w, T, first):
    shape = _shape(d, w, S=1 if T == 260 else 0)
    _run(shape, T, _sized_ids(T, shape.K, shape.E, first), 200 + T)


@pytest.mark.parametrize("d,w", [(64, 192), (960, 704)])
@pytest.mark.parametrize("rank", [0, 8])
def test_every_token_box(d, w, rank):
    """Segments whose tiles are 32, 64, .. 256 tokens wide in one launch: each of the eight boxes a half
    tile is fetched as, the last rows of a box belonging to the next segment, or past the end."""
    shape = _shape(d, w, E=12)
    first = [1, 40, 70, 100, 130, 165, 200, 230]
    _run(shape, 600, _sized_ids(600, 2, 12, first), 240, rank)


@pytest.mark.parametrize("d,w", [(64, 64), (320, 192), (512, 256)])
@pytest.mark.parametrize("rank", [8, 16])
def test_adapters(d, w, rank):
    """Adapters on some experts and on the shared one; with zero up matrices the plain forward's bits."""
    shape = _shape(d, w, E=6, S=1)
    T = 290
    args, _ = _run(shape, T, _sized_ids(T, 2, 6, [257, 33]), 210, rank)
    zero = []
    for e in range(shape.E):
        b = I.lora_block(210, shape, e, rank)
        for i, t in enumerate(I.split_lora(b, shape, rank)):
            if i % 2 == 1:
                t.zero_()
        zero.append(b.to(DEV))
    y0 = M.mcft_moe_forward_lora(*args, zero, [zero[0]], rank, 2.0)
    assert torch.equal(y0, M.mcft_moe_forward(*args))


def test_large_batches_of_unaligned_sizes_elsewhere():
    """d and w off the 256 / 128 multiples: the cached forward takes more than 64 tokens of them and its
    workspace serves mcft_gate_grad, and the no-allocation entry point serves batches whose workspace
    is larger than its static array, with the permuted activations in the outputs' memory (their bits
    against the plain forward's: test_gpu_same_bits.py)."""
    shape = _shape(320, 192, E=8, S=1)
    T, seed = 130, 220
    ids = _sized_ids(T, 2, 8, [40, 33])
    args, y = _run(shape, T, ids, seed)
    desc, x, idx, gate, experts, shared = args
    host = [b.pin_memory() for b in weights(shape, seed).experts]
    cache = M.mcft_cache_create(1, shape.E, 4, shape.expert_bytes, host, max_assign=T * shape.K)
    M.mcft_cache_step(cache, 0, idx)
    ws = torch.empty(M.mcft_moe_workspace_size(desc, T), dtype=torch.uint8, device=DEV)
    yc = M.mcft_moe_forward_cached(desc, x, idx, gate, cache, 0, shared, workspace=ws,
                                   copy_stream=torch.cuda.Stream())
    check_output(yc, f64(y), TOL_BF16, "cached forward")
    dy = I.hidden_iid(seed + 5, shape, T, tag="dy").to(DEV)
    dg = M.mcft_gate_grad(desc, dy, ws)
    ws2 = torch.empty_like(ws)
    M.mcft_moe_forward(*args, workspace=ws2)
    dg2 = M.mcft_gate_grad(desc, dy, ws2)
    M.mcft_device_error()
    assert ((dg - dg2).norm() / dg2.norm()).item() < 4 * 2.0 ** -8
    big = I.LayerShape("rows-noalloc", d=320, E=8, K=2, w=1728, n_shared=0, gate=I.GATE_RENORM,
                       dtype=I.BF16, cache_slots=4, keep=8)
    T = 1600  # 10.5 MiB of h and 3.9 of o fit the array; with 2 MiB of gathered rows they do not
    assert M.mcft_moe_workspace_size(M.desc_of(big), T) > 16 << 20
    ids = _sized_ids(T, 2, 8, [257])
    args, y = _run(big, T, ids, 230)
    yn = M.mcft_moe_forward_noalloc(*args)
    M.mcft_device_error()
    check_output(yn, f64(y), TOL_BF16, "no-allocation forward")

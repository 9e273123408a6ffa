"""The line between the one-CTA permutation (csrc/permute.cu) and the cluster's, for batches of more than 64
tokens: both sides of 1024 assignments against the oracle, on every path that follows (tensor cores with
and without padded segments, fp32), and the two sides' common rows bit for bit."""
import pytest
import torch

from paper_2609_34077_gb300 import inputs as I
from paper_2609_34077_gb300 import mcft as M
from tests.test_gpu_ffn_tile import _args
from tests.test_gpu_ffn_tile import _shape as _shape_f32
from tests.test_gpu_rows import _run, _shape, _sized_ids

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,S", [(4, 0), (64, 2)])
@pytest.mark.parametrize("T", [65, 511, 512, 513])
def test_sides_of_the_line(E, S, T):
    ids = _sized_ids(T, 2, E, [T, 7])
    args, y = _run(_shape(192, 128, E=E, S=S), T, ids, 280)
    big = [torch.cat([v, v, v]) for v in args[1:4]]  # over the line: the same tokens three times
    y3 = M.mcft_moe_forward(args[0], *big, *args[4:])
    M.mcft_device_error()
    assert torch.equal(y3, torch.cat([y, y, y]))


def test_padded_segments():
    """Two experts of 512 rows on average: the CTA-pair tiles, on the one-CTA permutation."""
    shape = I.LayerShape("permute-pair", d=256, E=2, K=1, w=128, n_shared=1, gate=I.GATE_RENORM, dtype=I.BF16,
                         cache_slots=1, keep=2)
    T = 1024
    args, y = _run(shape, T, _sized_ids(T, 1, 2, [300]), 281)
    M.mcft_set_tc_tiles(M.MCFT_TC_TILES_CTA_PAIR)
    try:
        yp = M.mcft_moe_forward(*args)
        M.mcft_device_error()
    finally:
        M.mcft_set_tc_tiles(M.MCFT_TC_TILES_ONE_CTA)
    assert torch.equal(yp, y)


@pytest.mark.parametrize("T", [512, 513])
def test_fp32(T):
    args, _ = _args(_shape_f32(128, 192, S=1), T, _sized_ids(T, 2, 4, [T, 7]), 282)
    y = M.mcft_moe_forward(*args)
    y2 = M.mcft_moe_forward(args[0], *[torch.cat([v, v, v]) for v in args[1:4]], *args[4:])
    M.mcft_device_error()
    assert torch.equal(y2[:T], y) and torch.equal(y2[T:2 * T], y)

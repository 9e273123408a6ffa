"""The SwiGLU epilogue of the tensor-core expert GEMMs over its whole range of gate values, seen bit by bit:
the layer's weights are chosen so that y = bf16(silu(g) * up) for a gate value g that is exact in fp32 (one
expert, gate weight one, W2 the identity). Around g = -87 to -89 the denominator 1 + e^-g passes 2^126 and
overflows; results down to 1e-37 are still bf16 numbers."""
import numpy as np
import pytest
import torch

from paper_2609_34077_gb300 import inputs as I
from paper_2609_34077_gb300 import mcft as M

pytestmark = pytest.mark.gpu
DEV = "cuda"
D, W = 256, 128


def _layer(dtype=torch.bfloat16):
    """Expert block with W1[j] = [1, b_j, 0...], W3[j] = [0, 0, 1, 0...], W2 the identity on W outputs."""
    b = (torch.arange(W) - W / 2) / 256.0  # exact in bf16
    w1, w3, w2 = torch.zeros(W, D), torch.zeros(W, D), torch.zeros(D, W)
    w1[:, 0], w1[:, 1], w3[:, 2] = 1.0, b, 1.0
    w2[:W] = torch.eye(W)
    blk = torch.cat([w1.reshape(-1), w3.reshape(-1), w2.reshape(-1)]).to(dtype)
    assert torch.equal(blk.float()[1::D][:W], b)
    return b, blk.to(DEV)


def _run(x0, up):
    """y [T, W] for gate values x0[t] + b[j] (x0 exact in bf16) and this up value."""
    b, blk = _layer()
    x = torch.zeros(len(x0), D)
    x[:, 0], x[:, 1], x[:, 2] = torch.from_numpy(x0), 1.0, up
    x = x.to(torch.bfloat16)
    assert torch.equal(x[:, 0].float(), torch.from_numpy(x0))
    desc = M.LayerDesc(D, 2, 1, W, 0, I.GATE_PLAIN, M.MCFT_BF16)
    idx = torch.zeros(len(x0), 1, dtype=torch.int32, device=DEV)
    gate = torch.ones(len(x0), 1, device=DEV)
    xd = x.to(DEV)
    y = M.mcft_moe_forward(desc, xd, idx, gate, [blk, blk])[:, :W].float().cpu().numpy()
    small = np.concatenate([M.mcft_moe_forward(desc, xd[i:i + 64].contiguous(), idx[i:i + 64], gate[i:i + 64],
                                               [blk, blk])[:, :W].float().cpu().numpy()
                            for i in range(0, len(x0), 64)])
    M.mcft_device_error()
    return x0[:, None].astype(np.float64) + b.numpy().astype(np.float64), y, small


def _gates(mode):
    if mode == "extremes":  # every quarter from -100 to -84, and the other end
        x0 = np.concatenate([np.arange(-100, -84, 0.5), np.arange(-70, -60, 0.5), [64.0, 88.0, 100.0, 1024.0]])
    else:
        x0 = np.arange(-64, 64, 0.25)
    return torch.from_numpy(x0).to(torch.bfloat16).float().numpy()


@pytest.mark.parametrize("mode,up", [("extremes", 1.0), ("extremes", 1024.0), ("middle", 1.0), ("middle", 0.75)])
@pytest.mark.parametrize("pair", [False, True])
def test_silu_over_its_range(mode, up, pair):
    x0 = _gates(mode)
    if pair:  # 512 rows an expert: the token-row tiles
        x0 = np.resize(x0, 1024)
        M.mcft_set_tc_tiles(M.MCFT_TC_TILES_CTA_PAIR)
    else:
        x0 = np.resize(x0, max(len(x0), 65))
    try:
        g, y, small = _run(x0, up)
    finally:
        M.mcft_set_tc_tiles(M.MCFT_TC_TILES_ONE_CTA)
    t = np.exp(-np.abs(g))
    ref = np.where(g < 0, g * t, g) / (1 + t) * up
    # fp32: e^-g within 2 units of the last place, sum, quotient (1) and product; then half a bf16 unit, 2^-8 of a
    # number just above a power of two. An
    # infinite 1 + e^-g (g < -88.73) makes the result zero; results under 2^-126 are rounded more coarsely.
    bound = np.abs(ref) * (2.0 ** -8 * 1.0001 + 6 * 2.0 ** -24) + 2.0 ** -133
    low = g < -88.72
    assert np.all(np.abs(y - ref)[~low] <= bound[~low])
    assert np.all(np.abs(y[low]) <= np.abs(ref[low]) * 1.01)
    # the decode kernels divide in IEEE fp32: a quotient one unit off crosses a bf16 boundary in 2^-15 of
    # the cases
    differ = np.mean(y != small)
    assert differ <= 2.0 ** -12, differ
    assert np.all(np.abs(y - small) <= 2.0 ** -7 * np.abs(small) * 1.0001)

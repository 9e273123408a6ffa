"""The middle vectors U = s A v of adapters keep fp32 accuracy on the tensor-core path of layers with d % 256
!= 0 or w % 128 != 0: the base product is made to cancel U's leading bits, so that the result is U's last one."""
import pytest
import torch

from paper_2609_34077_gb300 import inputs as I
from paper_2609_34077_gb300 import mcft as M

pytestmark = pytest.mark.gpu
DEV = "cuda"
C1, C2 = 37, 101  # columns in different slices of the down projection


def _forward(d, w, rank, T, m, which, value=None):
    """y[:, :w] = h of one adapted expert (W2 the identity), or with which = 2 o itself; A v is 1 + 2^-9 +
    2^-m in its first row, W v is -(1 + 2^-9) where A is adapted."""
    x = torch.zeros(T, d)
    x[:, 0], x[:, C1], x[:, C2] = 1.0, 2.0 ** -9, 2.0 ** -m
    if value is not None:
        x[3, C2] = value
    w1, w3, w2 = torch.zeros(w, d), torch.zeros(w, d), torch.zeros(d, w)
    a = [torch.zeros(rank, d), torch.zeros(rank, d), torch.zeros(rank, w)]
    b = [torch.zeros(w, rank), torch.zeros(w, rank), torch.zeros(d, rank)]
    sel = {1: 0, 3: 1, 2: 2}[which]
    a[sel][0, [0, C1, C2]] = 1.0
    b[sel][:, 0] = 1.0
    n = min(d, w)
    w2[:n, :n] = torch.eye(n)
    if which == 1:    # gate 2^-m, up 1
        w1[:, 0], w1[:, C1], w3[:, 0] = -1.0, -1.0, 1.0
    elif which == 3:  # gate 32 = silu(32), up 2^-m
        w1[:, 0], w3[:, 0], w3[:, C1] = 32.0, -1.0, -1.0
    else:             # h = 1, 2^-9 and 2^-m in columns 0, C1, C2
        w1[:, 0], w3[0, 0], w3[C1, C1], w3[C2, C2] = 32.0, 2.0 ** -5, 2.0 ** -5, 2.0 ** -5
        w2 = torch.zeros(d, w)
        w2[:, 0], w2[:, C1] = -1.0, -1.0
    blk = torch.cat([t.reshape(-1) for t in (w1, w3, w2)]).to(torch.bfloat16).to(DEV)
    ad = torch.cat([t.reshape(-1) for i in range(3) for t in (a[i], b[i])]).to(torch.bfloat16).to(DEV)
    desc = M.LayerDesc(d, 2, 1, w, 0, I.GATE_PLAIN, M.MCFT_BF16)
    idx = torch.zeros(T, 1, dtype=torch.int32, device=DEV)
    y = M.mcft_moe_forward_lora(desc, x.to(torch.bfloat16).to(DEV), idx, torch.ones(T, 1, device=DEV),
                                [blk, blk], [], [ad, None], [], rank, 1.0)
    M.mcft_device_error()
    return y[:, :n].float().cpu()


@pytest.mark.parametrize("d,w", [(192, 192), (256, 192), (320, 128)])
@pytest.mark.parametrize("rank", [8, 16])
@pytest.mark.parametrize("which,factor", [(1, 0.5), (3, 32.0), (2, 1.0)])
@pytest.mark.parametrize("T", [65, 300])
def test_last_bits_of_the_middle_vectors(d, w, rank, which, factor, T):
    for m in (12, 18, 22):
        y = _forward(d, w, rank, T, m, which)
        # exact but for silu(2^-m) = 2^-m (1 + 2^-m / 2) / 2 and bf16
        want = torch.full_like(y, factor * 2.0 ** -m)
        assert (y - want).abs().max() <= 2.0 ** -8 * want[0, 0], (m, y.min(), y.max())


@pytest.mark.parametrize("value", [float("inf"), float("nan"), 3.3895e38])
def test_middle_vectors_past_the_range_stay_in_their_row(value):
    """An infinite, undefined or nearly overflowing middle value: its token's outputs follow the decode
    kernels' (fp32 middle vectors) in being finite, the other tokens keep theirs."""
    y, ref = _forward(192, 192, 8, 70, 12, 2), _forward(192, 192, 8, 70, 12, 2, value)
    small = _forward(192, 192, 8, 8, 12, 2, value)
    assert torch.equal(torch.isfinite(ref[3]), torch.isfinite(small[3]))
    assert torch.equal(torch.cat([ref[:3], ref[4:]]), torch.cat([y[:3], y[4:]]))

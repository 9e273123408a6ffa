"""Entry points that promise mcft_moe_forward's results bit for bit, for bf16 layers whose sizes are no
multiples of 256 (d) and 128 (w) and batches of more than 64 tokens."""
import pytest
import torch

from paper_2609_34077_gb300 import inputs as I
from paper_2609_34077_gb300 import mcft as M
from tests.gpu_helpers import weights
from tests.test_gpu_rows import _run, _shape, _sized_ids

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("d,w,E,S,T", [(192, 192, 4, 0, 6300), (320, 1728, 8, 0, 1600), (128, 64, 8, 2, 5000),
                                       (192, 192, 4, 0, 65)])
def test_no_allocation_forward(d, w, E, S, T):
    """Batches whose permuted activations would not fit the static array, and a small one."""
    shape = _shape(d, w, E=E, S=S)
    args, _ = _run(shape, T, _sized_ids(T, 2, E, [65, 33]), 240)
    scratch = 16 << 20
    rows = T * (2 + S)
    assert T == 65 or rows * (4 * d + 2 * w) < scratch < M.mcft_moe_workspace_size(args[0], T)
    y = M.mcft_moe_forward_noalloc(*args)
    y2 = M.mcft_moe_forward_noalloc(*args)
    M.mcft_device_error()
    ref = M.mcft_moe_forward(*args)
    assert torch.equal(y, ref) and torch.equal(y2, ref)

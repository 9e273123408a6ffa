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


def _cached_step(cache, args, workspace=None, copy=None):
    M.mcft_cache_step(cache, 0, args[2])
    return M.mcft_moe_forward_cached(*args[:4], cache, 0, args[5], workspace=workspace,
                                     copy_stream=copy or torch.cuda.Stream())


@pytest.mark.parametrize("d,w,S", [(320, 192, 1), (64, 64, 0), (960, 704, 2), (256, 192, 0), (192, 128, 1)])
@pytest.mark.parametrize("T,first", [(65, [65, 1]), (130, [40, 33]), (700, [257, 256, 31])])
def test_cached_forward(d, w, S, T, first):
    """Misses into empty slots and staging buffers, then hits beside misses and bypassed experts; the
    workspaces serve the gate gradient alike."""
    E, B = 8, 3
    shape = _shape(d, w, E=E, S=S)
    host = [b.pin_memory() for b in weights(shape, 250).experts]
    cache = M.mcft_cache_create(1, E, B, shape.expert_bytes, host, max_assign=2 * T)
    dy = I.hidden_iid(255, shape, T, tag="dy").to(DEV)
    for step, sizes in enumerate((first, first[:1], first[::-1])):
        args, _ = _run(shape, T, _sized_ids(T, 2, E, sizes), 250)
        ws = torch.empty(M.mcft_moe_workspace_size(args[0], T), dtype=torch.uint8, device=DEV)
        yc = _cached_step(cache, args, ws)
        torch.cuda.synchronize()
        M.mcft_device_error()
        ws2 = torch.empty_like(ws)
        assert torch.equal(yc, M.mcft_moe_forward(*args, workspace=ws2)), step
        assert torch.equal(M.mcft_gate_grad(args[0], dy, ws), M.mcft_gate_grad(args[0], dy, ws2))


def test_cached_forward_under_capture():
    shape, T, E = _shape(192, 192, S=1), 90, 8
    args, _ = _run(shape, T, _sized_ids(T, 2, E, [33, 17]), 260)
    host = [b.pin_memory() for b in weights(shape, 260).experts]
    cache = M.mcft_cache_create(1, E, 4, shape.expert_bytes, host, max_assign=2 * T)
    ws = torch.empty(M.mcft_moe_workspace_size(args[0], T), dtype=torch.uint8, device=DEV)
    y, copy = torch.zeros_like(args[1]), torch.cuda.Stream()

    def step():
        M.mcft_cache_step(cache, 0, args[2])
        M.mcft_moe_forward_cached(*args[:4], cache, 0, args[5], y=y, workspace=ws, copy_stream=copy)

    step()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        step()
    y.zero_()
    g.replay()
    torch.cuda.synchronize()
    M.mcft_device_error()
    assert torch.equal(y, M.mcft_moe_forward(*args))


def test_cached_forward_of_an_expert_without_an_address_reports_it():
    """Ids that the cache step did not see have no block: the error word, and y stays as it was."""
    shape, T, E = _shape(192, 192), 70, 8
    args, _ = _run(shape, T, _sized_ids(T, 2, E, [33, 17]), 270)
    host = [b.pin_memory() for b in weights(shape, 270).experts]
    cache = M.mcft_cache_create(1, E, 4, shape.expert_bytes, host, max_assign=2 * T)
    M.mcft_cache_step(cache, 0, torch.zeros_like(args[2][:1, :1]))
    y = torch.full_like(args[1], 7.0)
    M.mcft_moe_forward_cached(*args[:4], cache, 0, args[5], y=y, copy_stream=torch.cuda.Stream())
    with pytest.raises(M.MCFTError):
        M.mcft_device_error()
    assert bool((y == 7.0).all())

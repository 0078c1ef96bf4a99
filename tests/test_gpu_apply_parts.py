"""gc_cache_apply where its split of the work changes: one part and several, fewer rows than a block, a
ragged last block, column tiles of at most 128 columns, row tiles whose second half is empty, more tiles
than CTA pairs; overwriting and adding.  The tolerance is that of the other tests of the call."""
import numpy as np
import pytest
import torch

from paper_2101_06983_b200 import inputs

from gpu_util import grad_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,d,d_in", [
    (3, 8, 64), (64, 264, 320), (65, 120, 384), (2113, 392, 128), (130, 2568, 2560), (4100, 256, 256),
])
def test_parts_and_tiles(oracle, rows, d, d_in):
    from paper_2101_06983_b200 import binding
    U = inputs.cache_rows(rows, d, seed=rows)
    bits, X = inputs.encoder_inputs(rows, d_in, seed=d)
    ref = oracle.cache_apply(U, X)
    dU = torch.from_numpy(U).cuda()
    dX = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda()
    need = binding.gc_cache_apply_workspace_bytes(rows, d, d_in)
    ws = torch.full((need + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    W = torch.full((d, d_in), float("nan"), device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.gc_cache_apply(dU, dX, W, False, ws[:need], st)
    once = W.clone()
    binding.gc_cache_apply(dU, dX, W, True, ws[:need], st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and bool((ws[need:] == 0xA5).all())
    assert grad_err(once.cpu().numpy(), ref) <= 1e-4
    assert grad_err(W.cpu().numpy(), 2 * ref) <= 1e-4


@pytest.mark.parametrize("planes", [0, 1, 2, 3])
def test_workspace_of_fewer_planes(oracle, planes):
    """256 bytes are enough for any call; what fits beside them is used, and nothing past it is written."""
    from paper_2101_06983_b200 import binding
    rows, d, d_in = 1000, 264, 320
    U = inputs.cache_rows(rows, d, seed=rows)
    bits, X = inputs.encoder_inputs(rows, d_in, seed=d)
    ref = oracle.cache_apply(U, X)
    dU = torch.from_numpy(U).cuda()
    dX = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda()
    need = max(256, planes * d * d_in * 4)
    assert need < binding.gc_cache_apply_workspace_bytes(rows, d, d_in)
    ws = torch.full((need + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    W = torch.full((d, d_in), float("nan"), device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.gc_cache_apply(dU, dX, W, False, ws[:need], st)
    once = W.clone()
    binding.gc_cache_apply(dU, dX, W, True, ws[:need], st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and bool((ws[need:] == 0xA5).all())
    assert grad_err(once.cpu().numpy(), ref) <= 1e-4
    assert grad_err(W.cpu().numpy(), 2 * ref) <= 1e-4
    with pytest.raises(binding.GradCacheError):
        binding.gc_cache_apply(dU, dX, W, True, ws[:255], st)

"""What a call through the binding meets outside the arithmetic: the device out of memory."""
import pytest
import torch

from paper_2506_15545_b200 import binding as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["forward", "forward_ex", "backward_ex", "prologue"])
def test_out_of_memory_is_torchs_own_error(call):
    """A result that torch has no room for: callers catch torch.OutOfMemoryError, free something and try again."""
    B, H, T, d = 1, 8, 16384, 128
    big = lambda *s: torch.empty(s, dtype=torch.bfloat16, device="cuda")
    q, k = big(B, H, T, d), big(B, 1, T, d)
    ws = R.alloc_workspace(q, k, 128, R.MODE_RATTN, R.FLAG_SAVE_RESIDUALS)
    calls = {"forward": lambda: R.rattn_forward(q, k, k, 128),
             "forward_ex": lambda: R.rattn_forward_ex(q, k, k, 128, workspace=ws),
             "backward_ex": lambda: R.rattn_backward_ex(q, k, k, q, 128, ws, flags=R.FLAG_SAVE_RESIDUALS),
             "prologue": lambda: R.rattn_qk_prologue(q, k)}
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (1 << 20)) / total)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            calls[call]()
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)

"""The first call of a process may fall into a stream capture: what the library sets up then must not break it."""
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

_PROGRAM = """
import sys
import torch
from paper_2506_15545_b200 import binding as R
gen = torch.Generator(device="cuda").manual_seed(3)
rnd = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()
T, w = 700, int(sys.argv[2])
q, k, v, g = rnd(1, 4, T, 128), rnd(1, 2, T, 128), rnd(1, 2, T, 128), rnd(1, 4, T, 128)
ws = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
kr, vr, st = rnd(1, 2, w, 128), rnd(1, 2, w, 128), torch.zeros(1, 2, 128, 128, device="cuda")
def step():
    if sys.argv[1] == "forward":
        return [R.rattn_forward(q, k, v, w)]
    if sys.argv[1] == "train":
        y = R.rattn_forward_ex(q, k, v, w, scale=0.1, workspace=ws, save_residuals=True)
        return [y, *R.rattn_backward_ex(q, k, v, g, w, ws, scale=0.1, flags=R.FLAG_SAVE_RESIDUALS)]
    x, z = R.rattn_qk_prologue(q[:, :, :1].contiguous(), k[:, :, :1].contiguous(), pos0=9)
    return [x, R.rattn_decode_step_ex(x.squeeze(2), z.squeeze(2), v[:, :, 0].contiguous(), kr.clone(), vr.clone(), st.clone(), 9)]
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    got = step()
graph.replay()
torch.cuda.synchronize()
assert all(torch.equal(a, b) for a, b in zip(got, step()))
print("same")
"""


@pytest.mark.parametrize("what,w", [("forward", 128), ("forward", 100), ("train", 128), ("decode", 128)])
def test_first_call_under_capture(what, w):
    r = subprocess.run([sys.executable, "-c", _PROGRAM, what, str(w)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stderr[-2000:]

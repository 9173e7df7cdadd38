"""The three ways the backward's reverse states are formed (a serial chain beside the dq kernel, terms formed in
parallel behind it, a chain on most of the SMs ahead of it), against the fp64 oracle: which one runs follows from
the sizes (tc_bwd.cu), so each case names one of them and an edge of it."""
import numpy as np
import pytest
import torch

from oracle import rattn_oracle as O
from paper_2506_15545_b200 import binding as R
from paper_2506_15545_b200 import workloads as W
from test_gpu_parity import GRAD_TOL, np64, rel_fro, small

pytestmark = pytest.mark.gpu

@pytest.mark.parametrize("B,Hq,Hkv,T,w,which", [
    (1, 4, 1, 385, 128, "terms: two"),
    (1, 8, 2, 769, 128, "terms: five, four parts of a group, the last query tile one row long"),
    (2, 2, 1, 1152, 256, "terms: six of a two-head group"),
    (1, 8, 8, 1024, 640, "chain beside dq: two steps, one head per group"),
    (5, 16, 16, 400, 128, "chain on more than half of the SMs"),
])
def test_reverse_states(B, Hq, Hkv, T, w, which):
    wl = small("rs", B, Hq, Hkv, T, 128, w, "bf16", 9300 + T, unit=True)
    q, k, v = W.make_qkv(wl)
    dy = W.make_dout(wl)
    qd, kd, vd, dyd = (t.cuda() for t in (q, k, v, dy))
    ws = R.alloc_workspace(qd, kd, w, R.MODE_RATTN, R.FLAG_SAVE_RESIDUALS)
    ws.fill_(0xff)                                     # nothing may be taken from a previous call's scratch
    R.rattn_forward_ex(qd, kd, vd, w, scale=wl.scale, workspace=ws, save_residuals=True)
    grads = R.rattn_backward_ex(qd, kd, vd, dyd, w, ws, scale=wl.scale, flags=R.FLAG_SAVE_RESIDUALS)
    again = R.rattn_backward_ex(qd, kd, vd, dyd, w, ws, scale=wl.scale, flags=R.FLAG_SAVE_RESIDUALS)
    torch.cuda.synchronize()
    assert R.rattn_read_status(ws) == 0

    for b in range(B if B < 5 else 1):                 # batch entries are alike: the wide case checks its first
        q1, k1, v1, dy1 = (np64(t[b:b + 1]) for t in (q, k, v, dy))
        want = O.backward(q1, k1, v1, dy1, w, wl.scale)
        for name, got, two, ref in zip(("dq", "dk", "dv"), grads, again, want[:3]):
            assert torch.equal(got, two), name
            assert np.isfinite(np64(got)).all(), name
            err = rel_fro(np64(got[b:b + 1]), ref)
            assert err <= GRAD_TOL, (which, name, err)
  

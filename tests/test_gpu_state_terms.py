"""The forward's chunk states formed as parallel terms and summed by a second kernel: long sequences on few K/V heads, fresh,
resumed and of different lengths, with the decode state, ahead of either forward kernel.  Rows are sampled, each against the
fp64 oracle; the kernels' names show that the path was taken."""
import numpy as np
import pytest
import torch

from oracle import rattn_oracle as O
from paper_2506_15545_b200 import binding as R
from paper_2506_15545_b200 import workloads as W
from test_gpu_full_size import sample_rows
from test_gpu_parity import TOL, np64, small

pytestmark = pytest.mark.gpu


def _buffers(B, w):
    ring = lambda: torch.full((B, 1, w, 128), 9.0, dtype=torch.bfloat16, device="cuda")
    return dict(state_out=torch.full((B, 1, 128, 128), 9.0, device="cuda"), k_ring_out=ring(), v_ring_out=ring())


def _call(*args, **kw):
    R.rattn_timing_enable(True)
    try:
        y = R.rattn_forward_ex(*args, **kw)
        torch.cuda.synchronize()
        assert "tc_state_sum" in R.rattn_timing_read()      # the terms' sum: the path this file is about
    finally:
        R.rattn_timing_enable(False)
    assert R.rattn_read_status(kw["workspace"]) == 0
    return y


def _check_rows(y, q, k, v, rows, w, scale, phi):
    """y, q [T,128] of one head, k, v [T,128]; rows: positions, y's are its last len(y)."""
    ref = O.forward_rows(np64(q), np64(k), np64(v), rows, w, scale, phi=phi)
    got = np64(y[torch.as_tensor(rows - (len(q) - len(y)), device=y.device)])
    err = np.abs(got - ref)
    bound = TOL["bf16"]["max_abs"] + 2.0 ** -8 * np.maximum(np.abs(ref) - 4.0, 0.0)   # beyond 4 the output's own spacing grows
    assert (err <= bound).all() and err.mean() <= TOL["bf16"]["mean_abs"], (err.max(), err.mean())


def _check_state(state, k, v, n, phi):
    ref = O.rla_state(np64(k), np64(v), max(0, n), phi)
    # phi(k) enters the tensor cores rounded to bf16 (2^-9 per term), the sums are fp32
    assert np.abs(np64(state) - ref).max() <= 2.0 ** -8 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("w,phi", [(512, R.PHI_SOFTMAX),      # single query tiles: every state is stored
                                   (1024, R.PHI_SOFTMAX),     # pairs: every second one
                                   (512, R.PHI_RELU)])
def test_fresh_sequence(w, phi):
    T = 8200                                                   # 65 chunks, the last one 8 tokens long
    wl = small("terms", 1, 8, 1, T, 128, w, "bf16", 9900 + w, unit=True)
    q, k, v = W.make_qkv(wl, "cuda")
    ws = R.alloc_workspace(q, k, w, R.MODE_RATTN, 0)
    ws.fill_(0xff)
    out = _buffers(1, w)
    y = _call(q, k, v, w, scale=wl.scale, workspace=ws, phi=phi, **out)
    for h in (0, 7):
        _check_rows(y[0, h], q[0, h], k[0, 0], v[0, 0], sample_rows(T, w, 24, h), w, wl.scale, phi)
    _check_state(out["state_out"][0, 0], k[0, 0], v[0, 0], T - w, phi)


@pytest.mark.parametrize("w", [512, 1024])
def test_resumed_sequence(w):
    first, T = 1500, 9800                                      # the chunk: 8300 tokens behind a history of w
    wl = small("termr", 1, 8, 1, T, 128, w, "bf16", 9950 + w, unit=True)
    q, k, v = W.make_qkv(wl, "cuda")
    cut = lambda a, b: (x[:, :, a:b].contiguous() for x in (q, k, v))
    out = _buffers(1, w)
    R.rattn_forward_ex(*cut(0, first), w, scale=wl.scale, workspace=R.alloc_workspace(q, k, w, R.MODE_RATTN, 0), **out)
    qc, kc, vc = cut(first, T)
    ws = R.alloc_workspace_chunked(qc, kc, w)
    ws.fill_(0xff)
    y = _call(qc, kc, vc, w, scale=wl.scale, workspace=ws, pos0=first, state_in=out["state_out"],
              k_ring_in=out["k_ring_out"], v_ring_in=out["v_ring_out"], **out)
    rows = sample_rows(T - first, w, 24, 3) + first
    for h in (0, 5):
        _check_rows(y[0, h], q[0, h], k[0, 0], v[0, 0], rows, w, wl.scale, R.PHI_SOFTMAX)
    _check_state(out["state_out"][0, 0], k[0, 0], v[0, 0], T - w, R.PHI_SOFTMAX)
    slots = torch.arange(T - w, T, device="cuda")
    assert torch.equal(out["k_ring_out"][0, 0, slots % w], k[0, 0, slots])


def test_entries_of_different_lengths():
    w, T, lens = 512, 8200, [8200, 3001, 400]
    wl = small("terml", 3, 8, 1, T, 128, w, "bf16", 9990, unit=True)
    q, k, v = W.make_qkv(wl, "cuda")
    ws = R.alloc_workspace(q, k, w, R.MODE_RATTN, 0)
    ws.fill_(0xff)
    out = _buffers(3, w)
    y = _call(q, k, v, w, scale=wl.scale, workspace=ws, seq_lens=torch.tensor(lens, dtype=torch.int32, device="cuda"), **out)
    for b, n in enumerate(lens):
        _check_rows(y[b, 2, :n], q[b, 2, :n], k[b, 0, :n], v[b, 0, :n], sample_rows(n, min(w, n - 1), 16, b), w, wl.scale, R.PHI_SOFTMAX)
        _check_state(out["state_out"][b, 0], k[b, 0], v[b, 0], n - w, R.PHI_SOFTMAX)

"""Failure detection on the device without faulting anything: every wait of the kernels is
bounded, and when one runs out the kernel stops by itself and leaves RATTN_ERR_TIMEOUT in the
workspace's status word.  The debug build of the library (librattn_dbg.so, include/rattn_debug.h)
can be told to withhold one mbarrier arrival -- a flag that nothing sets -- so that a wait does
run out; the test checks that the call returns, that the host reads the status, and that the
very next ordinary call on the same context is correct."""
import ctypes
import os

import numpy as np
import pytest
import torch

from oracle import rattn_oracle as O
from paper_2506_15545_b200 import binding as R
from paper_2506_15545_b200 import build as B
from paper_2506_15545_b200 import workloads as W
from test_gpu_parity import check, np64, small

pytestmark = pytest.mark.gpu

RATTN_ERR_TIMEOUT = -7


@pytest.fixture(scope="module")
def dbg():
    path = B.build(debug=True)
    L = ctypes.CDLL(path)
    vp, ci = ctypes.c_void_p, ctypes.c_int
    L.rattn_forward_ex.argtypes = [ctypes.POINTER(R.RattnParams), vp]
    L.rattn_forward_ex.restype = ci
    L.rattn_read_status.argtypes = [vp, vp]
    L.rattn_read_status.restype = ci
    L.rattn_debug_withhold_arrival.argtypes = [ci]
    L.rattn_debug_withhold_arrival.restype = ci
    yield L
    L.rattn_debug_withhold_arrival(0)


def _forward(L, q, k, v, out, ws, wl):
    p = R._params(q, k, v, out, wl.w, wl.scale, 1e-6, None, None, R.MODE_RATTN, ws, 0)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    return L.rattn_forward_ex(ctypes.byref(p), stream), stream


def test_expired_wait_is_reported_and_the_context_stays_usable(dbg):
    wl = small("fd", 1, 1, 1, 256, 128, 128, "bf16", 8100, unit=True)    # one work unit, one CTA
    assert R.rattn_uses_tensor_path(wl.d, wl.w)
    q, k, v = W.make_qkv(wl)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    ws = R.alloc_workspace(qd, kd, wl.w)
    out = torch.zeros_like(qd)

    dbg.rattn_debug_withhold_arrival(1)
    rc, stream = _forward(dbg, qd, kd, vd, out, ws, wl)
    assert rc == 0                                   # the launch itself is fine
    status = dbg.rattn_read_status(ctypes.c_void_p(ws.data_ptr()), stream)   # synchronises: the kernel has returned
    assert status == RATTN_ERR_TIMEOUT
    assert torch.cuda.current_stream().query()       # nothing left running

    # the switch off again: the same context, the same buffers, a correct result
    dbg.rattn_debug_withhold_arrival(0)
    rc, stream = _forward(dbg, qd, kd, vd, out, ws, wl)
    assert rc == 0
    assert dbg.rattn_read_status(ctypes.c_void_p(ws.data_ptr()), stream) == 0
    check(out, O.forward(np64(q), np64(k), np64(v), wl.w, wl.scale), "bf16", "after the time-out")
    # and the product library, loaded in the same process, is unaffected by the switch
    y = R.rattn_forward_ex(qd, kd, vd, wl.w, scale=wl.scale, workspace=ws)
    assert R.rattn_read_status(ws) == 0
    assert torch.equal(y, out)


def test_plain_forward_latches_its_status_before_freeing_its_scratch(dbg):
    """rattn_forward takes its scratch from the stream-ordered pool and frees it before it returns, so
    the status word in it is copied into the library first: rattn_forward_status reports the expired
    wait, is clear again afterwards, and the next call is correct."""
    vp, ci = ctypes.c_void_p, ctypes.c_int
    dbg.rattn_forward.argtypes = [vp, vp, vp, ci, ci, ci, ci, ci, ci, vp, vp]
    dbg.rattn_forward.restype = ci
    dbg.rattn_forward_status.argtypes = [vp]
    dbg.rattn_forward_status.restype = ci
    wl = small("fdp", 1, 1, 1, 256, 128, 128, "bf16", 8200, unit=True, scale=1.0)
    q, k, v = W.make_qkv(wl)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    out = torch.zeros_like(qd)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    call = lambda: dbg.rattn_forward(qd.data_ptr(), kd.data_ptr(), vd.data_ptr(), 1, 1, 1, wl.T, 128, wl.w,
                                     out.data_ptr(), stream)
    assert dbg.rattn_forward_status(stream) == 0
    dbg.rattn_debug_withhold_arrival(1)
    assert call() == 0
    assert dbg.rattn_forward_status(stream) == RATTN_ERR_TIMEOUT
    assert dbg.rattn_forward_status(stream) == 0          # reading clears it
    assert call() == 0
    dbg.rattn_debug_withhold_arrival(3)                   # the scratch cannot be given back: the expired wait is reported all the same
    assert dbg.rattn_forward_status(stream) == RATTN_ERR_TIMEOUT
    assert dbg.rattn_forward_status(stream) == -6         # RATTN_ERR_CUDA
    dbg.rattn_debug_withhold_arrival(0)
    assert call() == 0
    assert dbg.rattn_forward_status(stream) == 0
    check(out, O.forward(np64(q), np64(k), np64(v), wl.w, 1.0), "bf16", "after the time-out")
    # the product library's own word was never touched
    y = R.rattn_forward(qd, kd, vd, wl.w)
    assert R.rattn_forward_status() == 0 and torch.equal(y, out)


@pytest.mark.parametrize("B_,Hq,Hkv,T,w,mode", [
    (1, 2, 1, 384, 128, R.MODE_RATTN),          # single tiles behind a chain of states; all three backward kernels
    (1, 2, 2, 128, 128, R.MODE_RATTN),          # ... without states: the forward kernel alone, one tile
    (1, 2, 2, 700, 256, R.MODE_FULL_CAUSAL),    # the pair kernel
    (1, 40, 40, 1000, 128, R.MODE_RATTN),       # more units than CTAs hold at once: threads leave between two of them
])
def test_threads_that_share_a_barrier_leave_together(dbg, B_, Hq, Hkv, T, w, mode):
    """Some of the threads that meet at a named barrier (which has no bound) take a wait as run out that the others have
    passed: the kernel must end and report, not wait for those that left."""
    wl = small("fdb", B_, Hq, Hkv, T, 128, w, "bf16", 8300 + T, unit=True)
    q, k, v = (t.cuda() for t in W.make_qkv(wl))
    dy = W.make_dout(wl).cuda()
    ws = R.alloc_workspace(q, k, w, mode, R.FLAG_SAVE_RESIDUALS)
    out, dq, dk, dv = (torch.zeros_like(t) for t in (q, q, k, v))
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    dbg.rattn_backward_ex.argtypes = [ctypes.POINTER(R.RattnParams), ctypes.c_void_p]
    dbg.rattn_backward_ex.restype = ctypes.c_int
    p = R._params(q, k, v, out, w, wl.scale, 1e-6, None, None, mode, ws, R.FLAG_SAVE_RESIDUALS)
    p.dout, p.dq, p.dk, p.dv = (t.data_ptr() for t in (dy, dq, dk, dv))
    status = lambda: dbg.rattn_read_status(ctypes.c_void_p(ws.data_ptr()), stream)
    try:
        dbg.rattn_debug_withhold_arrival(2)
        assert dbg.rattn_forward_ex(ctypes.byref(p), stream) == 0
        assert status() == RATTN_ERR_TIMEOUT
        dbg.rattn_debug_withhold_arrival(0)
        assert dbg.rattn_forward_ex(ctypes.byref(p), stream) == 0 and status() == 0
        dbg.rattn_debug_withhold_arrival(2)
        assert dbg.rattn_backward_ex(ctypes.byref(p), stream) == 0
        assert status() == RATTN_ERR_TIMEOUT
    finally:
        dbg.rattn_debug_withhold_arrival(0)
    # the same context and buffers, normal operation: the product library's results
    assert dbg.rattn_forward_ex(ctypes.byref(p), stream) == 0
    assert dbg.rattn_backward_ex(ctypes.byref(p), stream) == 0
    assert status() == 0
    y = R.rattn_forward_ex(q, k, v, w, scale=wl.scale, mode=mode, workspace=ws, save_residuals=True)
    grads = R.rattn_backward_ex(q, k, v, dy, w, ws, scale=wl.scale, mode=mode, flags=R.FLAG_SAVE_RESIDUALS)
    assert all(torch.equal(a, b) for a, b in zip((out, dq, dk, dv), (y, *grads)))


@pytest.mark.parametrize("Hq,Hkv,T,w,train,handoff", [
    (2, 1, 384, 128, False, False),             # a chain of one step: nothing behind its only sum
    (2, 1, 384, 128, True, False),              # ... and the backward's
    (2, 2, 1000, 128, False, True),             # several steps, the last one for the decode state alone
    (8, 1, 8200, 512, False, True),             # terms formed in parallel
])
def test_a_chunk_state_that_gives_up_is_reported(dbg, Hq, Hkv, T, w, train, handoff):
    """The wait for a sum runs out in some threads of the chunk-state kernel and nowhere else: the status says so, also where
    no further step follows that could notice, and the sum does not leave."""
    gen = torch.Generator(device="cuda").manual_seed(13)
    rnd = lambda h: torch.randn(1, h, T, 128, generator=gen, device="cuda").bfloat16()
    q, k, v, dy = rnd(Hq), rnd(Hkv), rnd(Hkv), rnd(Hq)
    flags = R.FLAG_SAVE_RESIDUALS if train else 0
    ws = R.alloc_workspace(q, k, w, R.MODE_RATTN, flags)
    ws.fill_(0xAB)
    out, dq, dk, dv = (torch.zeros_like(t) for t in (q, q, k, v))
    state = torch.zeros(1, Hkv, 128, 128, device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    dbg.rattn_backward_ex.argtypes = [ctypes.POINTER(R.RattnParams), ctypes.c_void_p]
    p = R._params(q, k, v, out, w, 0.1, 1e-6, None, None, R.MODE_RATTN, ws, flags)
    p.dout, p.dq, p.dk, p.dv = (t.data_ptr() for t in (dy, dq, dk, dv))
    if handoff:
        p.state_out = state.data_ptr()
    status = lambda: dbg.rattn_read_status(ctypes.c_void_p(ws.data_ptr()), stream)
    try:
        dbg.rattn_debug_withhold_arrival(4)
        assert dbg.rattn_forward_ex(ctypes.byref(p), stream) == 0
        assert status() == RATTN_ERR_TIMEOUT
        if T == 384 and not train:
            assert (ws[512:] == 0xAB).all()     # behind the status block the chunk states: the only one has not been stored
        if train:
            dbg.rattn_debug_withhold_arrival(0)
            assert dbg.rattn_forward_ex(ctypes.byref(p), stream) == 0 and status() == 0
            dbg.rattn_debug_withhold_arrival(4)
            assert dbg.rattn_backward_ex(ctypes.byref(p), stream) == 0
            assert status() == RATTN_ERR_TIMEOUT
    finally:
        dbg.rattn_debug_withhold_arrival(0)
    assert dbg.rattn_forward_ex(ctypes.byref(p), stream) == 0 and status() == 0
    y = R.rattn_forward_ex(q, k, v, w, scale=0.1, workspace=ws, save_residuals=train, state_out=torch.empty_like(state) if handoff else None)
    assert torch.equal(out, y)


@pytest.mark.parametrize("B_,Hq,Hkv,w,pos", [
    (1, 8, 2, 512, 1000),        # cluster of 8 CTAs, the last of which gives up
    (40, 32, 8, 64, 100),        # one CTA per head
])
def test_a_decode_step_that_gives_up_writes_neither_output_nor_rings(dbg, B_, Hq, Hkv, w, pos):
    gen = torch.Generator(device="cuda").manual_seed(12)
    rnd = lambda *s, dt=torch.bfloat16: torch.randn(s, generator=gen, device="cuda").to(dt)
    q, k, v = rnd(B_, Hq, 128), rnd(B_, Hkv, 128), rnd(B_, Hkv, 128)
    cache = [rnd(B_, Hkv, w, 128), rnd(B_, Hkv, w, 128), rnd(B_, Hkv, 128, 128, dt=torch.float32)]
    out = torch.full_like(q, 7.0)
    vp = ctypes.c_void_p
    stream = vp(torch.cuda.current_stream().cuda_stream)
    dbg.rattn_decode_step_ex.argtypes = [ctypes.POINTER(R.RattnParams), vp, vp, vp, ctypes.c_int, vp]
    dbg.rattn_decode_status.argtypes = [vp]
    p = R._params(q, k, v, out, w, 0.1, 1e-6, None, None, R.MODE_RATTN, None, 0)
    step = lambda c: dbg.rattn_decode_step_ex(ctypes.byref(p), *(vp(t.data_ptr()) for t in c), pos, stream)
    assert dbg.rattn_decode_status(stream) == 0
    used = [t.clone() for t in cache]
    try:
        dbg.rattn_debug_withhold_arrival(2)
        assert step(used) == 0
        assert dbg.rattn_decode_status(stream) == RATTN_ERR_TIMEOUT
    finally:
        dbg.rattn_debug_withhold_arrival(0)
    assert torch.equal(used[0], cache[0]) and torch.equal(used[1], cache[1]) and (out == 7.0).all()
    # normal operation again: the product library's step
    used = [t.clone() for t in cache]
    assert step(used) == 0 and dbg.rattn_decode_status(stream) == 0
    y = R.rattn_decode_step_ex(q, k, v, *cache, pos, scale=0.1)
    assert torch.equal(y, out) and all(torch.equal(a, b) for a, b in zip(used, cache))

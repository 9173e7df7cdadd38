"""Kernel variants that are chosen by size, each side of every rule: clusters of 1 to 8 CTAs in the decode step, the
per-vector and the chunked prologue, single-tile and pair units of the tensor-core forward."""
import numpy as np
import pytest
import torch

from oracle import rattn_oracle as O
from paper_2506_15545_b200 import binding as R
from paper_2506_15545_b200 import workloads as W
from test_gpu_parity import check, np64, small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hkv,g,w,pos", [
    (1, 2, 4, 512, 1777),        # cluster of 8, one ring piece each
    (2, 8, 2, 448, 200),         # 8 CTAs, seven pieces' room, four with tokens: some CTAs have no slot at all
    (5, 8, 1, 64, 64),           # 4 CTAs on a single piece, exactly full
    (11, 8, 3, 128, 100),        # 2 CTAs, the last piece partly filled
    (19, 8, 8, 192, 1000),       # one CTA per head, an odd number of pieces
    (40, 4, 2, 64, 0),           # one CTA per head, no token yet
    (2, 8, 8, 512, 700),         # 8 heads a group, whose read-out takes the ring's place: clusters of 4, eight stages
    (9, 8, 7, 128, 500),         # ... 7 heads, two pieces: one CTA each
    (9, 8, 4, 512, 5000),        # 72 K/V heads: clusters of 4 would not all fit
    (12, 8, 4, 1024, 3000),      # 16 pieces: clusters of 2, two CTAs per SM
    (37, 8, 6, 192, 250),        # 296 heads, two CTAs per SM, four stages
])
def test_decode_clusters_against_the_portable_kernel(B, Hkv, g, w, pos):
    gen = torch.Generator(device="cuda").manual_seed(77 + B)
    rnd = lambda *s, dt=torch.bfloat16: torch.randn(s, generator=gen, device="cuda").to(dt)
    q, k, v = rnd(B, Hkv * g, 128), rnd(B, Hkv, 128), rnd(B, Hkv, 128)
    kr, vr, st = rnd(B, Hkv, w, 128), rnd(B, Hkv, w, 128), rnd(B, Hkv, 128, 128, dt=torch.float32)
    kr[:, :, min(pos, w):] = float("nan")              # slots that hold no token yet
    vr[:, :, min(pos, w):] = float("nan")
    other = [t.clone() for t in (kr, vr, st)]
    y = R.rattn_decode_step_ex(q, k, v, kr, vr, st, pos, scale=0.088)
    z = R.rattn_decode_step_ex(q, k, v, *other, pos, scale=0.088, flags=R.FLAG_FORCE_GENERIC)
    torch.cuda.synchronize()
    assert R.rattn_decode_status() == 0
    # both round y to bf16 once: one rounding step of values up to 8 in magnitude
    assert (y.float() - z.float()).abs().max().item() <= 2.0 ** -5
    assert (y.float() - z.float()).abs().mean().item() <= 5e-4
    assert torch.equal(kr.nan_to_num(), other[0].nan_to_num()) and torch.equal(vr.nan_to_num(), other[1].nan_to_num())
    # state: phi(k)^T v added in fp32 by both; phi from the fast exponential, 2^-21 relative per term of size up to 4
    assert (st - other[2]).abs().max().item() <= 1e-5


@pytest.mark.parametrize("layout", [R.LAYOUT_BHTD, R.LAYOUT_BTHD])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_prologue_per_vector_and_chunked_agree(layout, d, dtype):
    """4096 head vectors take the one kernel, 4160 the other; the shared tokens must come out alike."""
    gen = torch.Generator(device="cuda").manual_seed(5)
    B, Hq, Hkv, T = 1, 48, 16, 65                      # 65 tokens x 64 heads; the first 64 are 4096 vectors
    make = lambda H: torch.randn(B, T, H, d, generator=gen, device="cuda").to(dtype)
    q, k = make(Hq), make(Hkv)
    gain = torch.rand(d, generator=gen, device="cuda") + 0.5
    view = (lambda t: t) if layout == R.LAYOUT_BTHD else (lambda t: t.transpose(1, 2))
    call = lambda n: [view(t) for t in R.rattn_qk_prologue(view(q[:, :n]).contiguous(), view(k[:, :n]).contiguous(),
                                                            q_gain=gain, k_gain=gain, pos0=1000, layout=layout)]
    for a, b in zip(call(65), call(64)):
        a = a[:, :64].float()
        # the same fp32 arithmetic with sums in another order, rounded once
        assert (a - b.float()).abs().max().item() <= a.abs().max().item() * (2.0 ** -8 if dtype == torch.bfloat16 else 2e-6)
    assert R.rattn_qk_prologue_status() == 0


@pytest.mark.parametrize("B,Hq,Hkv,T,w", [
    (4, 18, 18, 384, 128),       # 216 tiles on two CTAs per SM
    (10, 16, 4, 300, 128),       # 480, the last of each head half empty, some CTAs taking two
    (1, 37, 37, 1000, 256),      # 296: one per CTA
    (1, 147, 49, 200, 128),      # 294
])
def test_forward_single_tiles_and_pairs(B, Hq, Hkv, T, w):
    wl = small("units", B, Hq, Hkv, T, 128, w, "bf16", 9500 + T, unit=True)
    q, k, v = W.make_qkv(wl)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    ws = R.alloc_workspace(qd, kd, w, R.MODE_RATTN, 0)
    ws.fill_(0xff)
    y = R.rattn_forward_ex(qd, kd, vd, w, scale=wl.scale, workspace=ws)
    torch.cuda.synchronize()
    assert R.rattn_read_status(ws) == 0
    g, heads = Hq // Hkv, sorted({0, Hq // 2, Hq - 1})
    for h in heads:
        ref = O.forward(np64(q[-1:, h:h + 1]), np64(k[-1:, h // g:h // g + 1]), np64(v[-1:, h // g:h // g + 1]), w, wl.scale)
        check(y[-1:, h:h + 1], ref, "bf16", f"head {h}")
    assert np.isfinite(np64(y)).all()


@pytest.mark.parametrize("B,Hq,Hkv,T,w,mode,train", [
    (1, 4, 1, 1100, 896, R.MODE_RATTN, False),     # the widest window of the single-tile kernel in inference
    (1, 4, 1, 1300, 1024, R.MODE_RATTN, False),    # ... pairs, the last one half empty
    (1, 4, 1, 1800, 1536, R.MODE_RATTN, True),     # ... single tiles in training
    (1, 4, 1, 1900, 1664, R.MODE_RATTN, True),     # ... pairs
    (1, 16, 4, 1400, 128, R.MODE_RATTN, False),    # 96 pairs, a chain of 9 steps: single tiles
    (1, 16, 4, 2200, 128, R.MODE_RATTN, False),    # 144 pairs, a chain of 16 steps that decides: pairs, one per CTA behind it
    (1, 16, 16, 2200, 128, R.MODE_RATTN, True),    # ... in training
    (1, 37, 37, 512, 128, R.MODE_SWA_ONLY, False),     # 148 tiles: one per SM
    (1, 37, 37, 513, 128, R.MODE_SWA_ONLY, False),     # 185 tiles: 111 pairs
    (2, 18, 9, 500, 128, R.MODE_FULL_CAUSAL, False),   # 144 tiles
    (1, 60, 20, 700, 128, R.MODE_FULL_CAUSAL, True),   # 360 tiles: 180 pairs, drawn from the counter
])
def test_forward_kernel_by_window_chain_and_mode(B, Hq, Hkv, T, w, mode, train):
    wl = small("rule", B, Hq, Hkv, T, 128, w, "bf16", 9400 + T, unit=True)
    q, k, v = W.make_qkv(wl)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    ws = R.alloc_workspace(qd, kd, w, mode, R.FLAG_SAVE_RESIDUALS if train else 0)
    ws.fill_(0xff)
    y = R.rattn_forward_ex(qd, kd, vd, w, scale=wl.scale, mode=mode, workspace=ws, save_residuals=train)
    torch.cuda.synchronize()
    assert R.rattn_read_status(ws) == 0
    g = Hq // Hkv
    for h in sorted({0, Hq // 2, Hq - 1}):
        ref = O.forward(np64(q[-1:, h:h + 1]), np64(k[-1:, h // g:h // g + 1]), np64(v[-1:, h // g:h // g + 1]), w, wl.scale,
                        mode=mode)
        check(y[-1:, h:h + 1], ref, "bf16", f"head {h}")
    assert np.isfinite(np64(y)).all()


def test_state_stride_knob():
    """m = 2 takes the pair kernel where single tiles would run: another kernel, the same operator."""
    wl = small("stride", 1, 8, 2, 1000, 128, 256, "bf16", 9450, unit=True)
    q, k, v = W.make_qkv(wl)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    ws = R.alloc_workspace(qd, kd, wl.w, R.MODE_RATTN, 0)
    out = {}
    try:
        for m in (0, 1, 2):
            R.rattn_tune(R.TUNE_STATE_STRIDE, m)
            ws.fill_(0xff)
            out[m] = R.rattn_forward_ex(qd, kd, vd, wl.w, scale=wl.scale, workspace=ws)
            assert R.rattn_read_status(ws) == 0
    finally:
        R.rattn_tune(R.TUNE_STATE_STRIDE, 0)
    assert torch.equal(out[0], out[1]) and not torch.equal(out[0], out[2])
    ref = O.forward(np64(q[:, 3:4]), np64(k[:, 0:1]), np64(v[:, 0:1]), wl.w, wl.scale)
    for y in out.values():
        check(y[:, 3:4], ref, "bf16")


@pytest.mark.parametrize("B,Hq,Hkv,T,w", [
    (8, 16, 16, 4096, 512),      # every key tile comes from HBM: loads in flight land out of order
    (1, 40, 8, 2048, 256),       # ... mostly from L2
])
def test_passes_over_the_same_inputs_are_bit_equal(B, Hq, Hkv, T, w):
    gen = torch.Generator(device="cuda").manual_seed(31)
    q, k, v, g = (torch.randn(B, H, T, 128, generator=gen, device="cuda").bfloat16() for H in (Hq, Hkv, Hkv, Hq))
    q, k = (x * torch.rsqrt(x.float().square().mean(-1, keepdim=True)).bfloat16() for x in (q, k))
    ws = R.alloc_workspace(q, k, w, R.MODE_RATTN, R.FLAG_SAVE_RESIDUALS)
    first = None
    for _ in range(60):
        y = R.rattn_forward_ex(q, k, v, w, scale=0.088, workspace=ws, save_residuals=True)
        out = (y, *R.rattn_backward_ex(q, k, v, g, w, ws, scale=0.088)[:3])
        first = first or out
        # no atomics on any of these: the order of every sum is fixed
        assert all(torch.equal(a, b) for a, b in zip(out, first))
    assert R.rattn_read_status(ws) == 0


@pytest.mark.parametrize("B,Hq,Hkv,T,d,w,dtype", [
    (1, 2, 2, 193, 64, 1, "f32"),        # window of two keys: every chunk but one through the states, last chunk one row
    (1, 2, 1, 320, 64, 63, "f32"),       # state boundary at a tile edge, group of two
    (2, 3, 1, 400, 128, 100, "bf16"),    # d = 128 in two slices, ragged, group of three
    (1, 40, 40, 256, 64, 64, "f32"),     # enough heads for tiles of 64 rows
    (1, 2, 2, 130, 64, 65, "f32"),       # a window that leaves no whole chunk
])
def test_portable_chunk_states(B, Hq, Hkv, T, d, w, dtype):
    wl = small("gst", B, Hq, Hkv, T, d, w, dtype, 9700 + T, unit=True)
    q, k, v = W.make_qkv(wl)
    dy = W.make_dout(wl)
    qd, kd, vd, dyd = (t.cuda() for t in (q, k, v, dy))
    ws = R.alloc_workspace(qd, kd, w, R.MODE_RATTN, R.FLAG_SAVE_RESIDUALS)
    ws.fill_(0xff)
    y = R.rattn_forward_ex(qd, kd, vd, w, scale=wl.scale, workspace=ws, save_residuals=True)
    grads = R.rattn_backward_ex(qd, kd, vd, dyd, w, ws, scale=wl.scale, flags=R.FLAG_SAVE_RESIDUALS)
    torch.cuda.synchronize()
    heads = slice(None) if Hq < 8 else slice(Hq - 1, Hq)          # a wide case checks its last head
    args = [np64(t[:, heads]) for t in (q, k, v)]
    check(y[:, heads], O.forward(*args, w, wl.scale), dtype, "forward")
    want = O.backward(*args, np64(dy[:, heads]), w, wl.scale)
    for name, got, ref in zip(("dq", "dk", "dv"), grads, want):
        got = np64(got[:, heads])
        assert np.linalg.norm(got - ref) <= (1e-4 if dtype == "f32" else 5e-2) * np.linalg.norm(ref), name


@pytest.mark.parametrize("Hq,Hkv,T,d,w,dtype", [
    (1, 1, 1024, 64, 1000, "f32"),       # portable kernels, dk/dv beside dq: its last key tiles are done first
    (2, 1, 700, 128, 500, "f32"),
    (2, 1, 700, 128, 256, "bf16"),       # tensor-core kernels
])
def test_gradients_in_place_of_the_inputs(Hq, Hkv, T, d, w, dtype):
    """dk, dv may be written over k, v and dq over dout: nothing reads those once the gradient is written."""
    wl = small("alias", 1, Hq, Hkv, T, d, w, dtype, 9800 + T, unit=True)
    q, k, v = (t.cuda() for t in W.make_qkv(wl))
    dy = W.make_dout(wl).cuda()
    ws = R.alloc_workspace(q, k, w, R.MODE_RATTN, R.FLAG_SAVE_RESIDUALS)
    R.rattn_forward_ex(q, k, v, w, scale=wl.scale, workspace=ws, save_residuals=True)
    apart = R.rattn_backward_ex(q, k, v, dy, w, ws, scale=wl.scale, flags=R.FLAG_SAVE_RESIDUALS)
    for _ in range(5):
        k2, v2, dy2 = k.clone(), v.clone(), dy.clone()
        R.rattn_backward_ex(q, k2, v2, dy2, w, ws, scale=wl.scale, flags=R.FLAG_SAVE_RESIDUALS, dq=dy2, dk=k2, dv=v2)
        assert all(torch.equal(a, b) for a, b in zip(apart, (dy2, k2, v2)))


@pytest.mark.parametrize("T,w,pos0", [(128, 512, 700), (512, 512, 512), (1000, 256, 3333), (300, 128, 1280)])
@pytest.mark.parametrize("place", ["apart", "in place", "shifted", "crossed"])
def test_rings_of_a_resumed_chunk(T, w, pos0, place):
    """The rings behind a chunk hold its tokens (and, of a chunk shorter than the window, older ones) wherever they are written:
    to memory of their own, over the incoming rings, over half of them, or each over the other's place."""
    gen = torch.Generator(device="cuda").manual_seed(T + w)
    B, Hq, Hkv, d = 2, 4, 2, 128
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    q, k, v = rnd(B, Hq, T, d), rnd(B, Hkv, T, d), rnd(B, Hkv, T, d)
    rings = [rnd(B, Hkv, w, d) for _ in range(2)]
    want = []
    for ring, x in zip(rings, (k, v)):
        r = ring.clone()
        for j in range(max(0, T - w), T):
            r[:, :, (pos0 + j) % w] = x[:, :, j]
        want.append(r)
    n = B * Hkv * w * d
    pool = torch.zeros(4 * n, device="cuda", dtype=torch.bfloat16)
    at = lambda i: pool[i:i + n].view(B, Hkv, w, d)
    k_in, v_in = at(0), at(n)
    k_in.copy_(rings[0])
    v_in.copy_(rings[1])
    k_out, v_out = {"apart": (at(2 * n), at(3 * n)), "in place": (k_in, v_in), "shifted": (at(n // 2), at(2 * n)),
                    "crossed": (v_in, k_in)}[place]
    state = torch.zeros(B, Hkv, d, d, device="cuda")
    ws = R.alloc_workspace_chunked(q, k, w)
    R.rattn_forward_ex(q, k, v, w, scale=0.1, workspace=ws, pos0=pos0, state_in=state, k_ring_in=k_in, v_ring_in=v_in,
                       state_out=torch.empty_like(state), k_ring_out=k_out, v_ring_out=v_out)
    assert R.rattn_read_status(ws) == 0
    assert torch.equal(k_out, want[0]) and torch.equal(v_out, want[1])


@pytest.mark.parametrize("T,lens", [(1, None), (77, None), (128, None), (116, [116, 1, 50])])
@pytest.mark.parametrize("w", [1024, 2048])
def test_prompts_of_one_tile_in_wide_windows(T, w, lens):
    """A prompt that every window covers: one operator whatever the window, and the same kernel as with a narrower one."""
    gen = torch.Generator(device="cuda").manual_seed(T)
    B = len(lens) if lens else 3
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    q, k, v = rnd(B, 8, T, 128), rnd(B, 2, T, 128), rnd(B, 2, T, 128)

    def run(w):
        ws = R.alloc_workspace(q, k, w, R.MODE_RATTN, 0)
        rings = [torch.empty(B, 2, w, 128, device="cuda", dtype=torch.bfloat16) for _ in range(2)]
        state = torch.full((B, 2, 128, 128), 7.0, device="cuda")
        more = dict(seq_lens=torch.tensor(lens, dtype=torch.int32, device="cuda")) if lens else {}
        out = R.rattn_forward_ex(q, k, v, w, scale=0.1, workspace=ws, state_out=state, k_ring_out=rings[0], v_ring_out=rings[1], **more)
        assert R.rattn_read_status(ws) == 0
        return [out[b, :, :n] for b, n in enumerate(lens or [T] * B)] + [r[:, :, :T] for r in rings] + [state]

    for x, y in zip(run(w), run(768)):
        assert torch.isfinite(x.float()).all() and torch.equal(x, y)


@pytest.mark.parametrize("B,Hq,Hkv,T,w", [
    (1, 2, 1, 700, 128),         # one head: a CTA alone
    (3, 2, 1, 700, 128),         # odd: a pair has a CTA without work
    (1, 14, 7, 1500, 256),
    (4, 8, 8, 900, 1024),        # nothing leaves the window but the decode state is formed
    (37, 1, 1, 300, 128),        # the most heads that go under the copy
    (38, 1, 1, 300, 128),        # behind it
    (1, 3, 3, 8200, 128),        # parallel terms: 3 x 64 CTAs
    (1, 5, 5, 8321, 1024),       # 5 x 58
])
def test_chain_under_the_hand_off(B, Hq, Hkv, T, w):
    """Behind the call's own copy the chunk states' CTAs are set up early and in pairs; without it the same kernel starts
    in full order: the same bits."""
    gen = torch.Generator(device="cuda").manual_seed(T + B)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    q, k, v = rnd(B, Hq, T, 128), rnd(B, Hkv, T, 128), rnd(B, Hkv, T, 128)
    ws = R.alloc_workspace(q, k, w, R.MODE_RATTN, 0)
    rings = dict(k_ring_out=torch.empty(B, Hkv, w, 128, device="cuda", dtype=torch.bfloat16))
    rings["v_ring_out"] = torch.empty_like(rings["k_ring_out"])
    got = []
    for more in ({}, rings, rings):
        ws.fill_(0xAB)
        state = torch.full((B, Hkv, 128, 128), 7.0, device="cuda")
        out = R.rattn_forward_ex(q, k, v, w, scale=0.1, workspace=ws, state_out=state, **more)
        assert R.rattn_read_status(ws) == 0
        got.append((out, state))
    for out, state in got[1:]:
        assert torch.isfinite(out.float()).all() and torch.equal(out, got[0][0]) and torch.equal(state, got[0][1])

"""Results whose every rounding is said in the kernels' source: fp32 sums of a fixed order, products fused or not.  The
restatements below round where the kernels do, so that what comes out has the same bits whatever the compiler or the number of
lanes on a row; library calls (exponential, reciprocal square root) are the same functions as in the kernels."""
import pytest
import torch

from paper_2506_15545_b200 import binding as R

pytestmark = pytest.mark.gpu


def fma(a, b, c):
    """a b + c, rounded once (the product is exact in fp64; the sum's rounding to fp64 is far below that to fp32)."""
    return (a.double() * b.double() + c.double()).float()


def phi_pair_sums(k):
    """The softmax map of bf16 rows: the halves' sums each in four interleaved chains, the first half's over the 16-byte chunks
    0 .. 7, the second half's over 4 .. 7, 0 .. 3."""
    l2e = torch.tensor(1.4426950408889634, device=k.device)
    x = k.float()
    m = x.amax(-1, keepdim=True)
    p = torch.exp2(fma(x, l2e, -(m * l2e)))
    half = []
    for lo, order in ((0, range(8)), (64, (4, 5, 6, 7, 0, 1, 2, 3))):
        cols = torch.cat([p[..., lo + 8 * c:lo + 8 * c + 8] for c in order], -1)
        s = torch.zeros_like(cols[..., :4])
        for i in range(0, 64, 4):
            s = s + cols[..., i:i + 4]
        half.append((s[..., 0] + s[..., 1]) + (s[..., 2] + s[..., 3]))
    return (p * (1 / (half[0] + half[1]))[..., None]).bfloat16()


@pytest.mark.parametrize("resumed", [False, True])
def test_feature_map_of_the_chunk_states(resumed):
    """Values that are unit vectors leave the mapped keys themselves in the state, behind a chain of one step."""
    g = torch.Generator(device="cuda").manual_seed(1)
    B, H, w, T = 4, 64, 128, 256
    q = torch.zeros(B, H, T, 128, device="cuda", dtype=torch.bfloat16)
    k = (2 * torch.randn(B, H, T, 128, generator=g, device="cuda")).bfloat16()
    v = torch.eye(128, device="cuda", dtype=torch.bfloat16).repeat(2, 1).expand(B, H, T, 128).contiguous()
    state = torch.empty(B, H, 128, 128, device="cuda")
    more, left = {}, k[:, :, :128]
    if resumed:                                          # the ring's keys leave, and those of the chunk's first tile
        ring = [k[:, :, 128:].contiguous(), v[:, :, 128:].contiguous()]
        more = dict(pos0=256, k_ring_in=ring[0], v_ring_in=ring[1], state_in=torch.zeros_like(state),
                    k_ring_out=torch.empty_like(ring[0]), v_ring_out=torch.empty_like(ring[1]))
        q, k, v = (t[:, :, :128].contiguous() for t in (q, k, v))
        left = ring[0]
        ws = R.alloc_workspace_chunked(q, k, w)
    else:
        ws = R.alloc_workspace(q, k, w)
    R.rattn_forward_ex(q, k, v, w, scale=0.1, workspace=ws, state_out=state, **more)
    assert R.rattn_read_status(ws) == 0
    assert torch.equal(state.transpose(-1, -2), phi_pair_sums(left).float())


def test_output_norm_gradient_with_gains():
    """Of a single token the window's weight is one: dv is the gradient that went through the norm and its gain."""
    g = torch.Generator(device="cuda").manual_seed(2)
    B, H, w = 256, 64, 128
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")
    q, k, dy = (rnd(B, H, 1, 128).bfloat16() for _ in range(3))
    v = (rnd(B, H, 1, 128) * 16).round() / 16            # the same in fp16
    v = v.bfloat16()
    v = torch.where(v.abs() < 1e-3, torch.full_like(v, 0.0625), v)
    gain = 1 + 0.1 * rnd(H, 128)
    ws = R.alloc_workspace(q, k, w, R.MODE_RATTN, R.FLAG_SAVE_RESIDUALS)
    more = dict(scale=0.1, workspace=ws, gamma_swa=gain, gamma_rla=torch.ones_like(gain))
    R.rattn_forward_ex(q, k, v, w, save_residuals=True, **more)
    _, _, dv = R.rattn_backward_ex(q, k, v, dy, w, flags=R.FLAG_SAVE_RESIDUALS, **more)
    assert R.rattn_read_status(ws) == 0

    o, gy = v.float()[:, :, 0], dy.float()[:, :, 0]
    t = gy * gain
    lanes = lambda x, half: x[..., 64 * half:64 * half + 64].unflatten(-1, (8, 8))
    ss = torch.zeros_like(lanes(o, 0)[..., 0])
    A = torch.zeros_like(ss)
    for e in range(8):
        lo, hi = lanes(o, 0)[..., e], lanes(o, 1)[..., e]
        ss = ss + fma(lo, lo, hi * hi)
        A = A + fma(lanes(t, 0)[..., e], lo, lanes(t, 1)[..., e] * hi)
    for step in (1, 2, 4):
        other = torch.arange(8, device="cuda") ^ step
        ss, A = ss + ss[..., other], A + A[..., other]
    ss, A = ss[..., :1], A[..., :1]
    full = lambda c: torch.full_like(ss, c)
    ir = torch.rsqrt(fma(ss, full(1 / 128), full(1e-6)))
    c = A * ir * ir * (1 / 128)
    want = (fma(gy, gain.expand_as(gy), -(o * c)) * ir).bfloat16()
    assert torch.equal(dv[:, :, 0], want)

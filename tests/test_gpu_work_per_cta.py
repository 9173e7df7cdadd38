"""Work that a persistent CTA does after its first piece: pairs of query tiles one behind the other, the rotation table of the
prologue refilled.  The arithmetic of a result does not depend on which CTA has it or what that CTA did before, so a few CTAs
with all of the work give the bits that many give."""
import numpy as np
import pytest
import torch

from oracle import rattn_oracle as O
from paper_2506_15545_b200 import binding as R
from test_gpu_full_size import sample_rows
from test_gpu_parity import TOL, np64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [1, 3])
@pytest.mark.parametrize("mode,T,w,lens", [
    (R.MODE_RATTN, 2300, 1024, None),                # nine pairs
    (R.MODE_RATTN, 2100, 1024, None),                # an odd number of tiles: a unit of one at the end
    (R.MODE_RATTN, 2400, 1024, [2400, 130, 1200]),   # units beyond an entry's end are passed over, some have a tile less
    (R.MODE_SWA_ONLY, 2600, 256, None),              # no residual part between the windows, an odd number of tiles
    (R.MODE_FULL_CAUSAL, 2600, 2600, None),
])
def test_pairs_one_behind_the_other(mode, T, w, lens, grid):
    """Scores of two tiles in one buffer, the next unit's behind the residual part that had its columns.  Without a residual
    branch the units are pairs only where there are more tiles than SMs."""
    g = torch.Generator(device="cuda").manual_seed(T + w)
    B = len(lens) if lens else 2
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    q, k, v = (rnd(B, h, T, 128).bfloat16() for h in (4, 2, 2))
    more = dict(scale=0.25, mode=mode, gamma_swa=1 + 0.1 * rnd(4, 128), gamma_rla=1 + 0.1 * rnd(4, 128))
    if lens:
        more["seq_lens"] = torch.tensor(lens, dtype=torch.int32, device="cuda")

    def run():
        ws = R.alloc_workspace(q, k, w)
        out = R.rattn_forward_ex(q, k, v, w, workspace=ws, **more)
        assert R.rattn_read_status(ws) == 0, "a device-side wait expired"
        return [out[b, :, :n] for b, n in enumerate(lens)] if lens else [out]

    assert mode == R.MODE_RATTN or (T + 127) // 128 * 4 * B > torch.cuda.get_device_properties(0).multi_processor_count
    many = run()
    prev = R.rattn_tune(R.TUNE_GRID, grid)
    try:
        few = run()
    finally:
        R.rattn_tune(R.TUNE_GRID, prev)
    for x, y in zip(many, few):
        assert torch.isfinite(x.float()).all() and torch.equal(x, y)
    if grid != 1:
        return
    for b, h in ((0, 0), (B - 1, 3)):                # ... and they are the right ones
        n = lens[b] if lens else T
        rows = sample_rows(n, min(w, n - 1), 24, T + h)
        ref = O.forward_rows(np64(q[b, h, :n]), np64(k[b, h // 2, :n]), np64(v[b, h // 2, :n]), rows, w, 0.25, mode=mode,
                             gamma_swa=np64(more["gamma_swa"][h]), gamma_rla=np64(more["gamma_rla"][h]))
        err = np.abs(np64(many[b][h] if lens else many[0][b, h])[rows] - ref)
        bound = TOL["bf16"]["max_abs"] + 2.0 ** -8 * np.maximum(np.abs(ref) - 4.0, 0.0)   # beyond 4 the output's own spacing grows
        assert (err <= bound).all() and err.mean() <= TOL["bf16"]["mean_abs"], (err.max(), err.mean())


@pytest.mark.parametrize("B,Hq,Hkv,T,d,dtype,entry_pos", [
    (1, 40, 8, 3000, 128, torch.bfloat16, False),    # a CTA's share of q: tens of positions
    (2, 3, 2, 7001, 128, torch.bfloat16, True),      # several refills, a batch entry's end inside a table
    (3, 2, 1, 9000, 64, torch.bfloat16, False),      # one head: more positions in a chunk than the usual table holds
    (700, 5, 3, 7, 128, torch.float32, True),        # many short entries
    (2500, 4, 1, 1, 64, torch.float32, True),        # one token each
])
def test_prologue_rotation_table(B, Hq, Hkv, T, d, dtype, entry_pos):
    """[B, T, H, d] takes sines and cosines from a table, [B, H, T, d] forms them per row: the same numbers."""
    g = torch.Generator(device="cuda").manual_seed(T + d)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").to(dtype)
    q, k, dq, dk = rnd(B, T, Hq, d), rnd(B, T, Hkv, d), rnd(B, T, Hq, d), rnd(B, T, Hkv, d)
    gains = dict(q_gain=1 + 0.1 * rnd(d).float(), k_gain=1 + 0.1 * rnd(d).float())
    if entry_pos:
        gains["pos"] = torch.randint(0, 100000, (B,), generator=g, device="cuda", dtype=torch.int32)
    t = lambda x: x.transpose(1, 2).contiguous()
    a = R.rattn_qk_prologue(q, k, layout=R.LAYOUT_BTHD, **gains)
    b = R.rattn_qk_prologue(t(q), t(k), **gains)
    for x, y in zip(a, b):
        assert torch.equal(t(x), y)
    a = R.rattn_qk_prologue_backward(q, k, dq, dk, layout=R.LAYOUT_BTHD, **gains)
    b = R.rattn_qk_prologue_backward(t(q), t(k), t(dq), t(dk), **gains)
    for x, y in zip(a[:2], b[:2]):
        assert torch.equal(t(x), y)
    for x, y in zip(a[2:], b[2:]):                   # fp32 sums of B T H terms in another order
        assert (x - y).abs().max() <= 1e-4 * y.abs().max()
    assert R.rattn_qk_prologue_status() == 0, "a device-side wait expired"

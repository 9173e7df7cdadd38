"""The work that users of the RAttention operator have it do, as measurable cases.

One pass is one attention layer's share of a larger step, taken through the public binding:
a decode step (qk-norm + rotary prologue, then the operator on the ring and the state), a
prefill (with the hand-off to decoding where a server takes it), or a training step (forward
with residuals, then backward).  Shapes are those of the paper's 3B and 12B layers (head size
128, 16/16, 32/8 and 40/8 heads, window 512), their neighbours, and the small fp32 layer that
numerics are checked on.  Positions, rings and states are a layer's at some point of a running
sequence; a pass does not move the position, because all layers of a model take a step at one.
"""
import math

import torch

from paper_2506_15545_b200 import binding as rb

# ---- the cases --------------------------------------------------------------------------
# kind "decode"   B tokens, one per sequence; per_entry: each sequence at a position of its own
# kind "prefill"  inference forward; handoff: state and rings go out to decoding; prologue: q, k
#                 pass qk-norm and rotary embedding first; chunk_at > 0: the T tokens resume a
#                 sequence at that position; ragged: a batch of prompts of different lengths;
#                 plain: the short entry point that takes no workspace (bf16, unit scale)
# kind "train"    forward with residuals + backward; mode "local" (window + linear branch) or
#                 "global" (full causal); layer: gains and their gradients, and the prologue and
#                 its backward around the operator; bthd: tensors as the projections leave them


def listed():
    return [
        # a single user's chat: one token, latency only
        _case("decode_single", "decode", B=1, H_q=32, H_kv=8, w=512, pos=1777),
        # a serving batch at the 12B layer's shape, every sequence at its own position
        _case("decode_batch32", "decode", B=32, H_q=32, H_kv=8, w=512, pos=32768, per_entry=True),
        # a short prompt that does not fill the window, of a length that fits no tile
        _case("prefill_short", "prefill", B=1, H_q=32, H_kv=8, T=333, w=512, handoff=True, prologue=True),
        # a server's batch of prompts of different lengths
        _case("prefill_ragged8", "prefill", B=8, H_q=32, H_kv=8, T=2048, w=512, handoff=True, ragged=True),
        # the next chunk of a long prompt
        _case("prefill_chunk", "prefill", B=2, H_q=32, H_kv=8, T=2048, w=512, handoff=True, chunk_at=6144),
        # the 3B layer's forward: scoring or evaluation, plain call
        _case("forward_3b", "prefill", B=4, H_q=16, H_kv=16, T=4096, w=512, plain=True),
        # long-context prefill at the 12B layer's shape
        _case("prefill_long", "prefill", B=8, H_q=32, H_kv=8, T=32768, w=512, handoff=True),
        # fine-tuning on one short sequence of odd length, small window
        _case("train_small", "train", B=1, H_q=16, H_kv=4, T=1111, w=128),
        # the 3B layer's training step
        _case("train_3b", "train", B=8, H_q=16, H_kv=16, T=4096, w=512),
        # the 12B layer's training step with grouped heads, gains, prologue and projection layout
        _case("train_12b_layer", "train", B=1, H_q=40, H_kv=8, T=8192, w=1024, layer=True, bthd=True),
        # the global layer that follows three local ones
        _case("train_global", "train", B=2, H_q=16, H_kv=16, T=4096, w=4096, mode="global"),
        # fp32 layer with heads of 64: numerics work, small models
        _case("train_fp32", "train", B=1, H_q=2, H_kv=2, T=1024, d=64, w=128, dtype="f32"),
    ]


_DEFAULTS = {
    "decode": dict(d=128, dtype="bf16", per_entry=False),
    "prefill": dict(d=128, dtype="bf16", handoff=False, prologue=False, ragged=False, chunk_at=0, plain=False,
                    bthd=False),
    "train": dict(d=128, dtype="bf16", mode="local", layer=False, bthd=False),
}


def _case(name, kind, **sizes):
    case = dict(_DEFAULTS[kind], kind=kind, **sizes)
    return dict(case, name=name) if name else case


# ---- more cases of the same ranges ---------------------------------------------------------
_HEADS = ((16, 16), (16, 4), (32, 8), (40, 8), (8, 8), (24, 8), (8, 1))
_MOST_FLOPS, _MOST_BYTES = 1.0e12, 2.0e9


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _draw_once(rng):
    H_q, H_kv = rng.choice(_HEADS)
    what = rng.choice(("decode", "decode", "prefill", "prefill", "chunk", "ragged", "train", "train", "global", "small"))
    w = 128 * _log(rng, 1, 16)
    if what == "decode":
        # caches that are not full yet, windows of whole 64-token pieces, batches up to a large server's
        w = 64 * _log(rng, 1, 32)
        return _case(None, "decode", B=_log(rng, 1, 128), H_q=H_q, H_kv=H_kv, w=w, pos=_log(rng, 16, 65536),
                     per_entry=rng.random() < 0.5)
    if what == "prefill":
        return _case(None, "prefill", B=_log(rng, 1, 16), H_q=H_q, H_kv=H_kv, T=_log(rng, 64, 32768), w=w,
                     handoff=rng.random() < 0.5, prologue=rng.random() < 0.3, bthd=rng.random() < 0.3)
    if what == "chunk":
        return _case(None, "prefill", B=_log(rng, 1, 8), H_q=H_q, H_kv=H_kv, T=_log(rng, 128, 8192), w=w,
                     handoff=True, chunk_at=w + _log(rng, 1, 32768))
    if what == "ragged":
        return _case(None, "prefill", B=rng.randint(2, 16), H_q=H_q, H_kv=H_kv, T=_log(rng, 256, 8192), w=w,
                     handoff=True, ragged=True)
    if what == "train":
        layer = rng.random() < 0.4
        return _case(None, "train", B=_log(rng, 1, 8), H_q=H_q, H_kv=H_kv, T=_log(rng, 256, 16384), w=w,
                     layer=layer, bthd=layer and rng.random() < 0.7)
    if what == "global":
        T = _log(rng, 256, 8192)
        return _case(None, "train", B=_log(rng, 1, 4), H_q=H_q, H_kv=H_kv, T=T, w=T, mode="global")
    # heads of 64, fp32, or windows of any length: small layers
    H_q, H_kv = rng.choice(((2, 2), (4, 2), (8, 2), (4, 4)))
    return _case(None, "train", B=rng.randint(1, 2), H_q=H_q, H_kv=H_kv, T=_log(rng, 100, 1500), w=_log(rng, 8, 512),
                 d=rng.choice((64, 64, 128)), dtype=rng.choice(("f32", "f32", "bf16")))


def draw(rng):
    while True:
        case = _draw_once(rng)
        need = work(case)
        if need["flops"] <= _MOST_FLOPS and need["bytes"] <= _MOST_BYTES:
            return case


# ---- inputs ---------------------------------------------------------------------------------
_DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


class _Inputs:
    """Seeded N(0,1) tensors on the GPU, optionally with rows of unit RMS (what qk-norm leaves)."""

    def __init__(self, case, seed):
        self.dtype = _DTYPES[case["dtype"]]
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def normal(self, *shape, dtype=None):
        return torch.randn(shape, generator=self.gen, device="cuda", dtype=dtype or self.dtype)

    def unit_rows(self, *shape):
        x = self.normal(*shape)
        for b in range(shape[0]):              # one batch entry at a time: bounded scratch at the long shapes
            row = x[b].float()
            x[b] = row * torch.rsqrt(row.square().mean(-1, keepdim=True))
        return x

    def gain(self, *shape):
        return 1.0 + 0.1 * self.normal(*shape, dtype=torch.float32)

    def cache(self, B, H_kv, w, d, tokens):
        """Rings and linear-attention state of sequences of `tokens` tokens so far."""
        k_ring, v_ring = self.unit_rows(B, H_kv, w, d), self.normal(B, H_kv, w, d)
        # sum of `left` outer products of a distribution over d features with a normal row
        left = max(0, tokens - w)
        state = self.normal(B, H_kv, d, d, dtype=torch.float32) * (1.6 * math.sqrt(left) / d)
        return k_ring, v_ring, state


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def run(state):
    return _RUN[state["kind"]](state)


def _shape(case, heads, tokens):
    B, d = case["B"], case["d"]
    return (B, tokens, heads, d) if case.get("bthd") else (B, heads, tokens, d)


def _lengths(case):
    """A ragged batch's prompt lengths: one of T tokens, which the batch is padded to, the others evenly in T/8 .. T."""
    B, T = case["B"], case["T"]
    return [T] + [int(T * (1 / 8 + 7 / 8 * (i + 0.5) / (B - 1))) for i in range(B - 1)]


# ---- decode -----------------------------------------------------------------------------------
def _prepare_decode(case, seed):
    x = _Inputs(case, seed)
    B, H_q, H_kv, d, w, pos = (case[n] for n in ("B", "H_q", "H_kv", "d", "w", "pos"))
    s = dict(kind="decode", scale=d ** -0.5, pos=pos, per_entry=case["per_entry"])
    s["q"], s["k"], s["v"] = x.normal(B, H_q, 1, d), x.normal(B, H_kv, 1, d), x.normal(B, H_kv, d)
    s["k_ring"], s["v_ring"], s["state"] = x.cache(B, H_kv, w, d, pos)
    s["q_gain"], s["k_gain"] = x.gain(d), x.gain(d)
    s["gamma_swa"], s["gamma_rla"] = x.gain(H_q, d), x.gain(H_q, d)
    # sequences that joined the batch at different times
    s["pos_dev"] = torch.randint(pos // 2, pos + 1, (B,), generator=x.gen, device="cuda", dtype=torch.int32) \
        if case["per_entry"] else None
    return s


def _run_decode(s):
    q, k = rb.rattn_qk_prologue(s["q"], s["k"], q_gain=s["q_gain"], k_gain=s["k_gain"], pos0=s["pos"],
                                pos=s["pos_dev"])
    out = rb.rattn_decode_step_ex(q.squeeze(2), k.squeeze(2), s["v"], s["k_ring"], s["v_ring"], s["state"], s["pos"],
                                  scale=s["scale"], gamma_swa=s["gamma_swa"], gamma_rla=s["gamma_rla"],
                                  pos_dev=s["pos_dev"])
    return out, s["k_ring"], s["v_ring"], s["state"]


# ---- prefill ------------------------------------------------------------------------------------
def _prepare_prefill(case, seed):
    x = _Inputs(case, seed)
    B, H_q, H_kv, T, d, w = (case[n] for n in ("B", "H_q", "H_kv", "T", "d", "w"))
    rows = x.normal if case["prologue"] else x.unit_rows
    s = dict(kind="prefill", w=w, scale=d ** -0.5, plain=case["plain"], prologue=case["prologue"])
    s["q"], s["k"] = rows(*_shape(case, H_q, T)), rows(*_shape(case, H_kv, T))
    s["v"] = x.normal(*_shape(case, H_kv, T))
    if case["plain"]:
        s["q"] *= s["scale"]                   # this entry point takes no scale: it is in the queries
        return s
    more = dict(layout=rb.LAYOUT_BTHD if case["bthd"] else rb.LAYOUT_BHTD)
    if case["chunk_at"]:
        more["k_ring_in"], more["v_ring_in"], more["state_in"] = x.cache(B, H_kv, w, d, case["chunk_at"])
        more["pos0"] = case["chunk_at"]
        more["workspace"] = rb.alloc_workspace_chunked(s["q"], s["k"], w)
    else:
        more["workspace"] = rb.alloc_workspace(s["q"], s["k"], w, rb.MODE_RATTN, 0, more["layout"])
    if case["prologue"]:
        s["q_gain"], s["k_gain"] = x.gain(d), x.gain(d)
    more["gamma_swa"], more["gamma_rla"] = x.gain(H_q, d), x.gain(H_q, d)
    if case["handoff"]:
        more["k_ring_out"] = torch.empty(B, H_kv, w, d, dtype=x.dtype, device="cuda")
        more["v_ring_out"] = torch.empty_like(more["k_ring_out"])
        more["state_out"] = torch.empty(B, H_kv, d, d, dtype=torch.float32, device="cuda")
    if case["ragged"]:
        lens = _lengths(case)
        order = torch.randperm(B, generator=torch.Generator().manual_seed(B + T)).tolist()
        lens = [lens[i] for i in order]
        more["seq_lens"] = torch.tensor(lens, dtype=torch.int32, device="cuda")
        # rows behind an entry's end are unspecified: the result is each entry's own rows
        more["out"] = torch.empty_like(s["q"])
        s["valid"] = [more["out"][b, :, :n] for b, n in enumerate(lens)]
    s["more"] = more
    return s


def _run_prefill(s):
    q, k = s["q"], s["k"]
    if s["plain"]:
        return rb.rattn_forward(q, k, s["v"], s["w"])
    more = s["more"]
    if s["prologue"]:
        q, k = rb.rattn_qk_prologue(q, k, q_gain=s["q_gain"], k_gain=s["k_gain"], layout=more["layout"])
    out = rb.rattn_forward_ex(q, k, s["v"], s["w"], scale=s["scale"], **more)
    return s.get("valid", out), more.get("k_ring_out"), more.get("v_ring_out"), more.get("state_out")


# ---- training -----------------------------------------------------------------------------------
def _prepare_train(case, seed):
    x = _Inputs(case, seed)
    H_q, H_kv, T, d, w = (case[n] for n in ("H_q", "H_kv", "T", "d", "w"))
    rows = x.normal if case["layer"] else x.unit_rows
    s = dict(kind="train", w=w, layer=case["layer"])
    s["q"], s["k"] = rows(*_shape(case, H_q, T)), rows(*_shape(case, H_kv, T))
    s["v"], s["dout"] = x.normal(*_shape(case, H_kv, T)), x.normal(*_shape(case, H_q, T))
    layout = rb.LAYOUT_BTHD if case["bthd"] else rb.LAYOUT_BHTD
    mode = rb.MODE_FULL_CAUSAL if case["mode"] == "global" else rb.MODE_RATTN
    s["more"] = dict(mode=mode, scale=d ** -0.5, layout=layout,
                     workspace=rb.alloc_workspace(s["q"], s["k"], w, mode, rb.FLAG_SAVE_RESIDUALS, layout))
    s["layout"] = layout
    s["gain_grads"] = {}
    if case["layer"]:
        s["q_gain"], s["k_gain"] = x.gain(d), x.gain(d)
        s["more"]["gamma_swa"], s["more"]["gamma_rla"] = x.gain(H_q, d), x.gain(H_q, d)
        s["gain_grads"] = dict(dgamma_swa=torch.empty(H_q, d, dtype=torch.float32, device="cuda"),
                               dgamma_rla=torch.empty(H_q, d, dtype=torch.float32, device="cuda"))
    return s


def _run_train(s):
    q, k, more = s["q"], s["k"], s["more"]
    if s["layer"]:
        q, k = rb.rattn_qk_prologue(q, k, q_gain=s["q_gain"], k_gain=s["k_gain"], layout=s["layout"])
    out = rb.rattn_forward_ex(q, k, s["v"], s["w"], save_residuals=True, **more)
    dq, dk, dv = rb.rattn_backward_ex(q, k, s["v"], s["dout"], s["w"], flags=rb.FLAG_SAVE_RESIDUALS,
                                      **more, **s["gain_grads"])
    if not s["layer"]:
        return out, dq, dk, dv
    dq, dk, dq_gain, dk_gain = rb.rattn_qk_prologue_backward(s["q"], s["k"], dq, dk, q_gain=s["q_gain"],
                                                             k_gain=s["k_gain"], layout=s["layout"])
    return out, dq, dk, dv, dq_gain, dk_gain, s["gain_grads"]["dgamma_swa"], s["gain_grads"]["dgamma_rla"]


_PREPARE = {"decode": _prepare_decode, "prefill": _prepare_prefill, "train": _prepare_train}
_RUN = {"decode": _run_decode, "prefill": _run_prefill, "train": _run_train}


# ---- what a pass cannot do without -----------------------------------------------------------------
def work(case):
    B, H_q, H_kv, d, w = (case[n] for n in ("B", "H_q", "H_kv", "d", "w"))
    elem = 4 if case["dtype"] == "f32" else 2
    ring, state = 2 * B * H_kv * w * d * elem, B * H_kv * d * d * 4
    if case["kind"] == "decode":
        # the ring read (one slot of it written), the state read and written, the token's vectors
        live = min(case["pos"], w)
        token = B * d * elem * (2 * H_q + 4 * H_kv)
        flops = B * (4 * d * (live + 1) * H_q + 2 * d * d * (H_q + H_kv))
        return {"bytes": 2 * B * H_kv * live * d * elem + 2 * state + token, "flops": flops}
    T = case["T"]
    q_bytes, kv_bytes = B * H_q * T * d * elem, B * H_kv * T * d * elem
    if case["kind"] == "prefill" and case["ragged"]:
        lens = _lengths(case)
        share = sum(lens) / (B * T)
    else:
        share, lens = 1.0, [T] * B
    before = min(case.get("chunk_at", 0), w)   # keys of the window that precede the chunk
    swa = rla = rla_kv = 0.0
    for n in lens:
        pairs = n * (w + 1) if before else n * min(n, w + 1) - min(n, w + 1) * (min(n, w + 1) - 1) / 2
        beyond = n if before else max(0, n - w - 1)
        swa += 2 * d * pairs * H_q
        rla += 2 * d * d * beyond * H_q
        rla_kv += 2 * d * d * beyond * H_kv
    if case.get("mode") == "global":
        rla = rla_kv = 0.0
    bytes_, flops = share * (2 * q_bytes + 2 * kv_bytes), 2 * swa + rla + rla_kv
    if case["kind"] == "prefill":
        if case["handoff"]:
            bytes_ += ring + state
        if before:
            bytes_ += ring + state
        return {"bytes": bytes_, "flops": flops}
    # backward: scores again and four products of the window branch; the linear branch's two products have two
    # gradients each; q, k, v, dout in and dq, dk, dv out
    flops += 5 * swa + 2 * rla + 2 * rla_kv
    return {"bytes": bytes_ + 3 * q_bytes + 4 * kv_bytes, "flops": flops}


def tolerance(case):
    # fp32: sums over up to T terms, gradients through two softmaxes and a norm; bf16: operands and results rounded
    # to 8 bits (2^-9 each), several in a row in the gradients
    return {"rel": 2e-5} if case["dtype"] == "f32" else {"rel": 1e-2}

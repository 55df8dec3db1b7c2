"""The work that programs have this package do, as cases that a timing harness can run.

A case is a dict of plain values.  ``listed()`` names the fixed ones, ``draw(rng)`` gives another one of the same ranges,
``prepare(case, seed)`` makes what a program holds before the call (inputs on the GPU and the workspaces, caches and
buffers it keeps), ``run(state)`` is one pass through the public entry points, ``work(case)`` what the pass cannot do
without and ``tolerance(case)`` how far another correct implementation may be from it.

Kinds of pass:

``train``    the operator's forward and backward through autograd (``path_attention``), o and every gradient out
``prefill``  a prompt: the forward for its outputs, then its key cache (``path_attn_fwd`` + ``path_attn_prefill_cache``)
``decode``   one decoding step over an in-place key cache (``path_attn_decode_step``)
``layer``    the layer front-end with its low-rank linear layer, forward and backward (``path_attn_lowrank_*``,
             ``path_attn_frontend_*``)
``ring``     the context-parallel forward, every rank's share played on this one GPU (``ring.virtual_ring_forward``)
``forward32``  the float32 forward that results are checked with (``path_attn_fwd`` on float32 tensors)
"""
from __future__ import annotations

import math

import torch

from paper_2505_16381_b200 import binding
from paper_2505_16381_b200.autograd import path_attention
from paper_2505_16381_b200.ring import GpuOps, virtual_ring_forward


# ------------------------------------------------------------------------------------------------------------- the cases

def _train(B, H, L, d, gate=False, retain=False):
    return {"kind": "train", "B": B, "H": H, "L": L, "d": d, "gate": gate, "retain": retain}


def _prefill(B, H, L, d, gate=False):
    return {"kind": "prefill", "B": B, "H": H, "L": L, "d": d, "gate": gate}


def _decode(B, H, t, d, gate=False):
    return {"kind": "decode", "B": B, "H": H, "t": t, "d": d, "gate": gate}


def _layer(B, H, L, d, D, r, gate=True):
    return {"kind": "layer", "B": B, "H": H, "L": L, "d": d, "D": D, "r": r, "gate": gate}


def _ring(B, H, L, d, segments, gate=False):
    return {"kind": "ring", "B": B, "H": H, "L": L, "d": d, "segments": segments, "gate": gate}


def _forward32(B, H, L, d, gate=False):
    return {"kind": "forward32", "B": B, "H": H, "L": L, "d": d, "gate": gate}


def listed():
    cases = [
        # a unit test, a toy model's layer: two heads, 256 tokens; launches and host work are everything
        ("train-tiny", _train(1, 2, 256, 64)),
        # a small language model's layer, head size 64, 2k context
        ("train-2k-d64", _train(8, 16, 2048, 64)),
        # the headline: one layer of a model of about 760M parameters at 4k context; the backward takes the forward's state
        ("train-4k-d128", _train(4, 16, 4096, 128, retain=True)),
        # PaTH-FoX at 8k context: the forget gate makes most far chunk pairs negligible
        ("train-8k-fox", _train(2, 16, 8192, 128, gate=True)),
        # packed documents: a length that is no multiple of the chunk, with the gate
        ("train-ragged-fox", _train(2, 8, 3001, 64, gate=True)),
        # long-context prompt
        ("prefill-32k", _prefill(1, 32, 32768, 128)),
        # a batch of chat-sized prompts of odd length, gated
        ("prefill-1500-fox", _prefill(4, 16, 1500, 64, gate=True)),
        # one token over a long cache, a single sequence
        ("decode-32k", _decode(1, 32, 32767, 128)),
        # one token for a batch of short conversations, gated
        ("decode-700-fox", _decode(8, 16, 700, 64, gate=True)),
        # the front-end at the paper's benchmark shape (batch 32, 32 heads of 64, 4k context), model width 2048, rank 64
        ("layer-4k", _layer(32, 32, 4096, 64, D=2048, r=64)),
        # the headline shape's forward with the sequence cut over four devices
        ("ring-4x1024", _ring(4, 16, 4096, 128, segments=4)),
        # the accuracy check in float32
        ("forward32-256", _forward32(1, 2, 256, 64)),
    ]
    return [dict(c, name=name) for name, c in cases]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def heads(most):   # batch x heads, at most `most` slices
        s = logint(1, max(1, most))
        h = min(s, rng.choice([1, 2, 3, 5, 8, 12, 16, 24, 32]))
        return max(1, s // h), h

    kind = rng.choice(["train", "train", "train", "prefill", "prefill", "decode", "decode", "layer", "ring", "forward32"])
    d, gate = rng.choice([64, 128]), rng.random() < 0.5
    if kind == "train":
        L = logint(64, 8192)
        L = L if rng.random() < 0.5 else max(128, L // 128 * 128)
        B, H = heads(min(256, (1 << 19) // L, (1 << 31) // (L * L)))
        return _train(B, H, L, d, gate, retain=rng.random() < 0.5)
    if kind == "prefill":
        L = logint(64, 32768)
        L = L if rng.random() < 0.5 else max(128, L // 128 * 128)
        B, H = heads(min(256, (1 << 19) // L, (1 << 35) // (L * L)))
        return _prefill(B, H, L, d, gate)
    if kind == "decode":
        t = logint(1, 65536)
        B, H = heads(min(1024, (1 << 21) // t))
        return _decode(B, H, t, d, gate)
    if kind == "layer":
        L, H = logint(64, 8192), rng.choice([4, 8, 12, 16, 24, 32])
        most = min(131072 // L, (1 << 28) // (H * d * L))
        return _layer(rng.randint(1, max(1, most)), H, L, d, D=rng.choice([512, 768, 1024, 1536, 2048]), r=rng.choice([64, 128]), gate=gate)
    if kind == "ring":
        segments = rng.randint(2, 8)
        L = max(64 * segments, logint(512, 8192))
        B, H = heads(min(64, (1 << 18) // L))
        return _ring(B, H, L, d, segments, gate)
    return _forward32(rng.randint(1, 2), rng.randint(1, 4), logint(32, 512), d, gate)


# ------------------------------------------------------------------------------------------------------ inputs and passes

def _operator_inputs(gen, B, H, L, d, gate, dtype=torch.bfloat16):
    """q, k ~ N(0,1)/sqrt(d), v ~ N(0,1), w of unit norm, beta = 2 sigmoid(N(0,1)), log f = logsigmoid(N(0,1) + 3)."""
    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    q, k = ((normal(B, H, L, d) / d ** 0.5).to(dtype) for _ in range(2))
    v = normal(B, H, L, d).to(dtype)
    w = torch.nn.functional.normalize(normal(B, H, L, d), dim=-1).to(dtype)
    beta = 2.0 * torch.sigmoid(normal(B, H, L))
    log_f = torch.nn.functional.logsigmoid(normal(B, H, L) + 3.0) if gate else None
    return q, k, v, w, beta, log_f


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind, B, H, d, gate = case["kind"], case["B"], case["H"], case["d"], case["gate"]
    state = dict(case)
    if kind == "train":
        inputs = _operator_inputs(gen, B, H, case["L"], d, gate)
        state["inputs"] = [None if t is None else t.requires_grad_() for t in inputs]
        state["d_o"] = torch.randn(B, H, case["L"], d, generator=gen, device="cuda").to(torch.bfloat16)
    elif kind == "prefill":
        q = _operator_inputs(gen, B, H, case["L"], d, gate)
        state["inputs"] = q
        state["workspace"] = binding.alloc_workspace(q[0], gate, False)
        state["cache"] = binding.alloc_cache(B, H, case["L"] + 128, d, gate)     # room for the answer's first tokens
    elif kind == "decode":
        t, cap = case["t"], case["t"] + 128
        cache = binding.alloc_cache(B, H, cap, d, gate)
        cache["kc"][:, :, :t] = torch.randn(B, H, t, d, generator=gen, device="cuda") / d ** 0.5
        cache["vc"][:, :, :t] = torch.randn(B, H, t, d, generator=gen, device="cuda").to(torch.bfloat16)
        if gate:
            log_f = torch.nn.functional.logsigmoid(torch.randn(B, H, t, generator=gen, device="cuda") + 3.0)
            cache["gc"][:, :, :t] = log_f.cumsum(-1)
        state["cache"] = cache
        state["workspace"] = binding.decode_workspace(B, H, cap, d)
        token = _operator_inputs(gen, B, H, 1, d, gate)
        state["token"] = [None if x is None else x[:, :, 0].contiguous() for x in token]
    elif kind == "layer":
        L, D, r, C = case["L"], case["D"], case["r"], H * d

        def normal(*shape):
            return torch.randn(*shape, generator=gen, device="cuda")

        state["x"] = normal(B, L, D).to(torch.bfloat16)
        state["w1"] = (normal(r, D) / D ** 0.5).to(torch.bfloat16)
        state["w2"] = (normal(C, r) / r ** 0.5).to(torch.bfloat16)
        state["conv_w"] = normal(C, 3) / 3 ** 0.5
        state["beta_logit"] = normal(B, L, H)
        state["gate_logit"] = normal(B, L, H) + 3.0 if gate else None
        state["dw"] = normal(B, H, L, d).to(torch.bfloat16)
        state["dbeta"] = normal(B, H, L)
        state["dlog_f"] = normal(B, H, L) if gate else None
    elif kind == "ring":
        L, n = case["L"], case["segments"]
        q, k, v, w, beta, log_f = _operator_inputs(gen, B, H, L, d, gate)
        ends = [L * i // n for i in range(n + 1)]
        state["segments"] = [
            {name: None if x is None else x[:, :, a:b].contiguous()
             for name, x in zip(("q", "k", "v", "w", "beta", "log_f"), (q, k, v, w, beta, log_f))}
            for a, b in zip(ends, ends[1:])]
        state["ops"] = GpuOps(B, H, d, has_gate=gate)
    elif kind == "forward32":
        inputs = _operator_inputs(gen, B, H, case["L"], d, gate, torch.float32)
        state["inputs"] = inputs
        state["workspace"] = binding.alloc_workspace(inputs[0], gate, False)
    else:
        raise ValueError(kind)
    return state


def run(state):
    kind = state["kind"]
    if kind == "train":
        o = path_attention(*state["inputs"], retain_state=state["retain"])
        wanted = [t for t in state["inputs"] if t is not None]
        return [o.detach(), *torch.autograd.grad(o, wanted, state["d_o"])]
    if kind == "prefill":
        q, k, v, w, beta, log_f = state["inputs"]
        o, lse = binding.path_attn_fwd(q, k, v, w, beta, log_f, workspace=state["workspace"])
        binding.path_attn_prefill_cache(k, v, w, beta, state["cache"], log_f, workspace=state["workspace"])
        return [o, lse, state["cache"]]
    if kind == "decode":
        q, k, v, w, beta, log_f = state["token"]
        o, lse = binding.path_attn_decode_step(q, k, v, w, beta, state["cache"], state["t"], log_f,
                                               workspace=state["workspace"])
        return [o, lse, state["cache"]]
    if kind == "layer":
        H = state["H"]
        z, t = binding.path_attn_lowrank_fwd(state["x"], state["w1"], state["w2"])
        w, beta, log_f = binding.path_attn_frontend_fwd(z, state["conv_w"], state["beta_logit"], state["gate_logit"], H=H)
        dz, dconv_w, dbeta_logit, dgate_logit = binding.path_attn_frontend_bwd(
            z, state["conv_w"], state["beta_logit"], state["dw"], state["dbeta"], state["gate_logit"], state["dlog_f"], H=H)
        dx, dw1, dw2 = binding.path_attn_lowrank_bwd(state["x"], state["w1"], state["w2"], t, dz)
        return [w, beta, log_f, dx, dw1, dw2, dconv_w, dbeta_logit, dgate_logit]
    if kind == "ring":
        return [list(r) for r in virtual_ring_forward(state["ops"], state["segments"])]
    q, k, v, w, beta, log_f = state["inputs"]
    return list(binding.path_attn_fwd(q, k, v, w, beta, log_f, workspace=state["workspace"]))


# ------------------------------------------------------------------------------------------------------------ the measure

# keys back at which the workloads' gate (-0.07 a token on average) has decayed to e^-30
_GATE_REACH = 430


def _pairs(L, gate):
    """Causal (query, key) pairs that count: all, or those the gate leaves above e^-30."""
    n = min(L, _GATE_REACH) if gate else L
    return n * (n + 1) // 2 + (L - n) * n


def work(case):
    kind, B, H, d, gate = case["kind"], case["B"], case["H"], case["d"], case["gate"]
    S = B * H
    if kind == "decode":
        t = case["t"]
        # cached keys read and written (float32), values read (bf16), gate prefix read; the token's own vectors
        per_token = 8 * d + 2 * d + (4 if gate else 0)
        return {"bytes": S * (t * per_token + 16 * d), "flops": S * t * 8.0 * d}
    if kind == "layer":
        M, D, r, C, g = B * case["L"], case["D"], case["r"], H * d, 2 if gate else 1
        # x, dw, the weights and the logits in; w, dx, the gates and all gradients out
        elems16 = M * D + 2 * r * (D + C) + M * C * 2 + M * D
        return {"bytes": 2 * elems16 + 4 * M * H * g * 4, "flops": 6.0 * M * r * (D + C)}
    L = case["L"]
    rows, pairs = S * L, S * _pairs(L, gate)
    vec = rows * (2 if gate else 1) * 4                    # beta and log f
    if kind == "train":                                    # q k v w dO in, o dq dk dv dw out; two products forward, five backward
        return {"bytes": 10 * rows * d * 2 + 2 * vec, "flops": 14.0 * pairs * d}
    if kind == "prefill":                                  # q k v w in, o lse and the cache out
        return {"bytes": 5 * rows * d * 2 + rows * (4 * d + 2 * d + 4) + 2 * vec, "flops": 4.0 * pairs * d}
    if kind == "ring":
        return {"bytes": 5 * rows * d * 2 + vec + 4 * rows, "flops": 4.0 * pairs * d}
    return {"bytes": 5 * rows * d * 4 + vec + 4 * rows, "flops": 4.0 * pairs * d}


def tolerance(case):
    # Against the same formulas in float64 (L = 256 ... 2048, both head sizes): o 2.2e-3, gradients 4.6e-3 (dw; bf16 operands
    # of chained products), cached keys 1.7e-3, decoded o 1.7e-3, the front-end's bf16 outputs 3.0e-3, float32 forward 2.2e-6.
    return {"train": {"rel": 2e-2}, "prefill": {"rel": 1e-2}, "decode": {"rel": 4e-3}, "layer": {"rel": 8e-3},
            "ring": {"rel": 1e-2}, "forward32": {"rel": 1e-5}}[case["kind"]]

"""The layer's work as a program that uses it has it done: inputs, one pass, and what a pass must cost.

Every case goes through the methods of ``arl2.Layer`` (the C entry points, one to one).  The sizes are
those of the workload table (one latent frame = 1560 tokens, a block of one or three frames, 12 heads
of dimension 128 in the base model, 40 in the wider one, up to 8 streams served together) and ragged
ones between them.
"""
from __future__ import annotations

import math

import torch

from paper_2605_16579_b200 import arl2, workload

_BF16_OPS = ("step", "clean", "commit", "delta", "decay", "tokens", "module", "teacher", "token_level")


def _case(name, op, B, H, L, dtype="bf16", D=128, cache=0, gate="head"):
    return {"name": name, "op": op, "B": B, "H": H, "L": L, "D": D, "dtype": dtype, "cache": cache, "gate": gate}


def listed():
    return [
        # the smallest call: a 16 x 16 latent frame in the fp32 mode, where launches and latency count
        _case("step_tiny_fp32", "step", 1, 2, 256, dtype="fp32", D=64),
        # one denoise pass over a one-frame block of the base model (interactive generation)
        _case("step_frame", "step", 1, 12, 1560),
        # several streams of an odd block length, as a server with mixed resolutions sees them
        _case("step_ragged", "step", 3, 12, 1001),
        # one denoise pass over a three-frame block of the wider model: four of these per block
        _case("step_wide", "step", 1, 40, 4680),
        # the clean pass of eight streams served together: output and state update in one call
        _case("clean_serving", "clean", 8, 12, 4680),
        # the state update of a one-frame block of the base model
        _case("commit_frame", "commit", 1, 12, 1560),
        # the state update of a three-frame block of the wider model
        _case("commit_wide", "commit", 1, 40, 4680),
        # the state update with the delta rule, a three-frame block of the base model
        _case("delta_block", "delta", 1, 12, 4680),
        # the state update token by token with per-token gates, the same block
        _case("tokens_block", "tokens", 1, 12, 4680),
        # the whole attention module (projections, core, output projection) of the base model
        _case("module_block", "module", 1, 12, 4680),
        # a softmax layer of the stack: the block's queries over a cache of four blocks
        _case("teacher_cache", "teacher", 1, 12, 4680, cache=4 * 4680),
        # the comparison mode in which each token reads its own state, a one-frame block
        _case("token_level_frame", "token_level", 1, 12, 1560),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    largest = max(work(c)["flops"] for c in listed())
    while True:
        op = rng.choice(_BF16_OPS + ("step",))
        H = rng.choice((2, 5, 8, 12, 16, 24, 40))
        B = rng.choice((1, 1, 1, 2, 3, 4, 8))
        L = _log_int(rng, 200, 4680)
        dtype, D, cache, gate = "bf16", 128, 0, "head"
        if op == "teacher":
            cache = L * rng.randint(1, 4) + rng.choice((0, 0, 17))
        if op in ("step", "commit") and rng.random() < 0.2:
            dtype, D, H, L = "fp32", rng.choice((64, 128)), rng.choice((2, 4, 12)), _log_int(rng, 200, 1560)
        elif op == "step":
            gate = rng.choice(("head", "head", "scalar", "element"))
        c = _case("", op, B, H, L, dtype, D, cache, gate)
        del c["name"]
        # fp32 work runs on the FMA units: counted against the same ceiling at a thirtieth of the rate
        if work(c)["flops"] * (30 if dtype == "fp32" else 1) <= largest:
            return c


# ------------------------------------------------------------------------------------------ inputs
def _device():
    return "cuda:0" if torch.cuda.is_available() else "cpu"


def _inputs(case, seed):
    """Everything that a pass reads, on the device and in the dtypes the layer takes."""
    B, H, L, D, op = case["B"], case["H"], case["L"], case["D"], case["op"]
    dev = _device()
    dt = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))

    def randn(*shape, std=1.0, mean=0.0, dtype=torch.float32):
        return (torch.randn(*shape, generator=gen, device=dev) * std + mean).to(dtype)

    x = {}
    if op == "module":
        d = H * D
        x["x"] = randn(B, L, d, dtype=dt)
        for n in ("w_q", "w_k", "w_v", "w_o"):
            x[n] = randn(d, d, std=d ** -0.5, dtype=dt)
        x["w_g"] = randn(d, H, std=0.1 * d ** -0.5, dtype=dt)
    else:
        lk = case["cache"] if op == "teacher" else L
        if op in ("step", "clean", "teacher", "token_level"):
            x["q"] = randn(B, L, H, D, dtype=dt)
        x["k"] = randn(B, lk, H, D, dtype=dt)
        x["v"] = randn(B, lk, H, D, dtype=dt)
        if op in ("step", "clean", "token_level"):
            gshape = {"head": (B, L, H), "scalar": (B, L), "element": (B, L, H, D)}[case["gate"]]
            x["gate"] = randn(*gshape, std=0.1)
    if op in ("clean", "commit", "delta"):
        x["decay"] = randn(B, H, mean=3.0, std=0.5)
    if op in ("decay", "tokens", "token_level"):
        x["alpha"] = randn(B, L, H, mean=7.0)
    if op == "tokens":
        x["beta"] = randn(B, L, H)
    if op == "delta":
        # rates at which a pass repeated on the same block contracts: mean rate x L / D stays near 1
        x["beta"] = randn(B, L, H, mean=-4.0)
    if op != "teacher":
        eye = torch.eye(D, device=dev)
        for n in ("wq", "wk", "wv"):
            x[n] = (eye + randn(H, D, D, std=0.02)).to(dt)
        cos, sin = workload.rope_tables(L, D)
        x["cos"], x["sin"] = cos.to(dev), sin.to(dev)
        # a state of the size that the update rule settles at
        s_std = 1.0 if op == "tokens" else math.sqrt(L / D) * 3.0
        x["state"] = randn(B, H, D, D, std=s_std)
    return x


_GATE_FLAGS = {"head": 0, "scalar": arl2.ARL2_FLAG_GATE_SCALAR, "element": arl2.ARL2_FLAG_GATE_ELEMENTWISE}


def prepare(case, seed):
    B, H, L, D, op = case["B"], case["H"], case["L"], case["D"], case["op"]
    x = _inputs(case, seed)
    flags = _GATE_FLAGS[case["gate"]] | (arl2.ARL2_FLAG_TOKEN_GATES if op == "tokens" else 0)
    layer = arl2.Layer(B, H, L, D, case["dtype"], device=_device(), flags=flags)
    if op != "teacher":
        layer.set_params(x["wq"], x["wk"], x["wv"], x["cos"], x["sin"])
        layer.set_state(x["state"])
    st = {"op": op, "layer": layer, "x": x}
    shape = (B, L, H, D)
    if op in ("step", "clean", "teacher", "token_level", "module"):
        st["out"] = torch.empty(shape, dtype=layer.dtype, device=layer.device)
    if op == "module":
        layer.set_projections(x["w_q"], x["w_k"], x["w_v"], x["w_g"], x["w_o"])
        for n in ("q", "k", "v"):
            st[n] = torch.empty(shape, dtype=layer.dtype, device=layer.device)
        st["g"] = torch.empty(B, L, H, dtype=torch.float32, device=layer.device)
        st["y"] = torch.empty(B, L, H * D, dtype=layer.dtype, device=layer.device)
    return st


def run(state):
    op, layer, x = state["op"], state["layer"], state["x"]
    if op == "step":
        return layer.denoise_step(x["q"], x["k"], x["v"], x["gate"], out=state["out"])
    if op == "clean":
        out = layer.clean_pass(x["q"], x["k"], x["v"], x["gate"], x["decay"], out=state["out"])
        return out, layer.state
    if op == "commit":
        layer.commit(x["k"], x["v"], x["decay"])
        return layer.state
    if op == "delta":
        layer.commit_delta(x["k"], x["v"], x["decay"], x["beta"])
        return layer.state
    if op == "decay":
        layer.commit_decay_tokens(x["k"], x["v"], x["alpha"])
        return layer.state
    if op == "tokens":
        layer.commit_tokens(x["k"], x["v"], x["alpha"], x["beta"])
        return layer.state
    if op == "teacher":
        return layer.teacher_step(x["q"], x["k"], x["v"], out=state["out"])
    if op == "token_level":
        return layer.denoise_step_token_level(x["q"], x["k"], x["v"], x["gate"], x["alpha"], out=state["out"])
    assert op == "module"
    q, k, v, g = layer.project_in(x["x"], state["q"], state["k"], state["v"], state["g"])
    o = layer.denoise_step(q, k, v, g, out=state["out"])
    return layer.project_out(o, state["y"])


# -------------------------------------------------------------------------------------------- work
def work(case):
    B, H, L, D, op = case["B"], case["H"], case["L"], case["D"], case["op"]
    e = 4 if case["dtype"] == "fp32" else 2
    bh, t = B * H, B * H * L * D
    lk = case["cache"] if op == "teacher" else L
    maps = H * D * D * e
    rope = L * D * 4
    gate = 4 * {"head": bh * L, "scalar": B * L, "element": t}[case["gate"]]
    attend = 4 * bh * L * lk * D
    read = 4 * bh * L * D * D            # Q W and Q' S
    update = 4 * bh * L * D * D          # K W and K'^T V (the value map may be applied after the sum)
    s = bh * D * D * 4
    if op == "step":
        return {"bytes": 4 * t * e + gate + s + maps + rope, "flops": attend + read}
    if op == "clean":
        return {"bytes": 4 * t * e + gate + 2 * s + 3 * maps + rope, "flops": attend + read + update}
    if op == "commit":
        return {"bytes": 2 * t * e + 2 * s + 2 * maps + rope, "flops": update}
    if op == "decay":
        return {"bytes": 2 * t * e + 4 * bh * L + 2 * s + 2 * maps + rope, "flops": update}
    if op == "delta":
        return {"bytes": 2 * t * e + 4 * bh * L + 2 * s + 2 * maps + rope, "flops": update + 2 * bh * L * D * D}
    if op == "tokens":
        return {"bytes": 2 * t * e + 8 * bh * L + 2 * s + 2 * maps + rope, "flops": update + 4 * bh * L * D * D}
    if op == "teacher":
        return {"bytes": 2 * t * e + 2 * B * H * lk * D * e, "flops": attend}
    if op == "token_level":
        return {"bytes": 4 * t * e + 8 * bh * L + s + 3 * maps + rope, "flops": attend + read + update}
    assert op == "module"
    d = H * D
    proj = 2 * B * L * d * (4 * d + H)
    return {"bytes": 2 * B * L * d * e + d * (4 * d + H) * e + s + maps + rope, "flops": attend + read + proj}


def tolerance(case):
    # about four times the distance from the 64-bit result that was measured: fp32 2e-7 (other summation
    # orders reach a little further), softmax over a cache 2.4e-3, step and clean pass 2.9e-3, module 3.7e-3,
    # token by token 4e-3, state after a gated-linear commit 6e-4, after the delta rule 6.8e-3 (its two terms
    # nearly cancel)
    if case["dtype"] == "fp32":
        return {"rel": 2e-6}
    return {"rel": {"commit": 3e-3, "decay": 3e-3, "teacher": 1e-2, "step": 1.2e-2, "clean": 1.2e-2,
                    "token_level": 1.2e-2, "module": 1.5e-2, "tokens": 1.6e-2, "delta": 2.7e-2}[case["op"]]}


# ------------------------------------------------------------------------------------------- exact
def _rope64(x, cos, sin):
    """x [..., L, D] with adjacent pairs rotated by the tables [L, D/2]."""
    c, s = cos.double(), sin.double()
    x0, x1 = x[..., 0::2], x[..., 1::2]
    return torch.stack((x0 * c - x1 * s, x0 * s + x1 * c), dim=-1).flatten(-2)


def _phi64(x, w, cos, sin, eps=1e-6):
    """L2Norm(RoPE(x W)) for x [B, H, L, D], w [H, D, D]."""
    u = _rope64(torch.matmul(x, w.double()), cos, sin)
    return u / torch.sqrt((u * u).sum(-1, keepdim=True) + eps)


def _attend64(q, k, v):
    out = torch.empty_like(q)
    scale = q.shape[-1] ** -0.5
    for b in range(q.shape[0]):
        for h in range(q.shape[1]):
            for r in range(0, q.shape[2], 2048):
                p = torch.softmax(q[b, h, r:r + 2048] @ k[b, h].T * scale, dim=-1)
                out[b, h, r:r + 2048] = p @ v[b, h]
    return out


def _heads64(x):
    return x.double().permute(0, 2, 1, 3).contiguous()


def exact(case, seed):
    B, H, L, D, op = case["B"], case["H"], case["L"], case["D"], case["op"]
    if not torch.cuda.is_available() and work(case)["flops"] > 2e10:
        return None
    x = _inputs(case, seed)
    if op == "teacher":
        return _attend64(_heads64(x["q"]), _heads64(x["k"]), _heads64(x["v"])).permute(0, 2, 1, 3).contiguous()
    cos, sin, S = x["cos"], x["sin"], x["state"].double()
    if op == "module":
        xs = x["x"].double()
        q, k, v = (torch.matmul(xs, x[n].double()).view(B, L, H, D).permute(0, 2, 1, 3).contiguous()
                   for n in ("w_q", "w_k", "w_v"))
        gate = torch.matmul(xs, x["w_g"].double())
    else:
        q = _heads64(x["q"]) if "q" in x else None
        k, v = _heads64(x["k"]), _heads64(x["v"])
        gate = x["gate"].double() if "gate" in x else None
    if gate is not None:   # -> [B, H, L, 1 or D]
        gate = torch.sigmoid(gate)
        gate = {"head": lambda g: g.permute(0, 2, 1).unsqueeze(-1), "scalar": lambda g: g.view(B, 1, L, 1),
                "element": lambda g: g.permute(0, 2, 1, 3)}[case["gate"]](gate)
    out = None
    if op in ("step", "clean", "module", "token_level"):
        o = _attend64(_rope64(q, cos, sin), _rope64(k, cos, sin), v)
        qf = _phi64(q, x["wq"], cos, sin)
        if op != "token_level":
            o = o + gate * torch.matmul(qf, S)
        out = o
    if op in ("clean", "commit", "delta", "decay", "tokens", "token_level"):
        kf = _phi64(k, x["wk"], cos, sin)
        vf = torch.matmul(v, x["wv"].double())
    if op in ("clean", "commit"):
        S = torch.sigmoid(x["decay"].double())[..., None, None] * S + kf.transpose(-1, -2) @ vf
    if op == "delta":
        beta = torch.sigmoid(x["beta"].double()).permute(0, 2, 1).unsqueeze(-1)
        S = torch.sigmoid(x["decay"].double())[..., None, None] * S + kf.transpose(-1, -2) @ (beta * (vf - kf @ S))
    if op in ("decay", "tokens", "token_level"):
        alpha = torch.sigmoid(x["alpha"].double()).permute(0, 2, 1)   # [B, H, L]
        beta = torch.sigmoid(x["beta"].double()).permute(0, 2, 1) if op == "tokens" else None
        read = torch.empty_like(v) if op == "token_level" else None
        for i in range(L):
            ki, vi, ai = kf[:, :, i], vf[:, :, i], alpha[:, :, i, None, None]
            if read is not None:
                read[:, :, i] = torch.matmul(qf[:, :, i].unsqueeze(-2), S).squeeze(-2)
            if beta is not None:
                vi = beta[:, :, i, None] * (vi - torch.matmul(ki.unsqueeze(-2), S).squeeze(-2))
            S = ai * S + ki.unsqueeze(-1) * vi.unsqueeze(-2)
        if read is not None:
            out = out + gate * read
    if out is not None:
        out = out.permute(0, 2, 1, 3).contiguous()
    if op == "module":
        return torch.matmul(out.view(B, L, H * D), x["w_o"].double())
    if op == "clean":
        return out, S
    return S if out is None else out

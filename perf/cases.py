"""What this framework is timed on: the calls that programs make of it, from one decode step to a
long training sequence.

A case names an entry point (``op``) and its sizes.  ``prepare`` makes what a program holds before
the call (tokens, states, the scratch workspace), ``run`` makes the call, ``exact`` computes the
same results with plain torch in 64 bits, and ``work`` counts the bytes and operations that the
call cannot do without.

Inputs follow the recipe of the repository's workloads: query and key rows of unit length drawn
from a Gaussian, values N(0, 1).  A normalised call divides by a sum of products of queries and
keys, which is used with nonnegative features so that the sum stays away from zero; its queries
and keys are the absolute values of such rows.  Decode states are those of a short prompt.
"""
from __future__ import annotations

import math

import torch

from paper_2510_27258_gb300 import hla

EPS = 1e-6
PROMPT = 64  # tokens of the prompt that decode states and continued prefills start from
TILE = 128   # tokens per step of the 64-bit recurrences

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(op, B, H, n, d, dv, dtype, **flags):
    c = {"op": op, "B": B, "H": H, "n": n, "d": d, "dv": dv, "dtype": dtype, "masked": True, "normalized": False,
         "state_in": False, "state_out": False}
    c.update(flags)
    return c


def listed():
    return [
        # one sequence being decoded interactively: the smallest call, launch and latency bound
        _case("step", 1, 16, 1, 64, 64, "bf16", name="decode_one"),
        # a serving batch's decode step on the paper's state tuple (the repository's decode workload)
        _case("step", 64, 32, 1, 128, 128, "bf16", name="decode_batch"),
        # a decode step of the asymmetric operator for a small batch
        _case("ahla_step", 8, 32, 1, 128, 128, "bf16", name="ahla_decode"),
        # the forward of a training step at head size 64 (the repository's middle workload)
        _case("forward", 8, 16, 2048, 64, 64, "bf16", name="train_forward"),
        # long sequences, normalised output, head size 128 (the headline workload)
        _case("forward", 2, 16, 16384, 128, 128, "bf16", normalized=True, name="long_normalized"),
        # the prompt of one request, of no particular length, whose final state the decode steps go on from
        _case("forward", 1, 32, 1999, 128, 128, "bf16", state_out=True, name="prefill"),
        # a single-precision model: small batch, ragged length
        _case("forward", 2, 16, 1000, 64, 64, "f32", name="forward_f32"),
        # the gradients of a training step at head size 64
        _case("backward", 8, 16, 2048, 64, 64, "bf16", name="train_backward"),
        # the gradients of the normalised operator at head size 128, as the long workload would be trained
        _case("backward", 2, 16, 4096, 128, 128, "bf16", normalized=True, name="train_backward_d128"),
        # the asymmetric operator's training forward (the repository's workload)
        _case("ahla", 8, 16, 2048, 64, 64, "bf16", name="ahla_forward"),
        # the asymmetric operator's prefill: ragged prompt, final state kept for decoding
        _case("ahla", 1, 32, 1999, 128, 128, "bf16", state_out=True, name="ahla_prefill"),
        # the third-order forward in single precision (the repository's workload)
        _case("hla3", 4, 8, 4096, 32, 32, "f32", name="third_order"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """A case of the same ranges: every entry point, head sizes 16 to 128, short to long and ragged
    sequences, few to many heads, both token types, outputs plain and normalised, with and without states."""
    op = rng.choice(["step", "step_sde", "ahla_step", "forward", "forward", "forward", "backward", "backward", "ahla",
                     "hla3"])
    if op in ("step", "step_sde", "ahla_step"):
        d = rng.choice([64, 128, 128])
        return _case(op, _log_int(rng, 1, 64), rng.choice([8, 16, 24, 32]), 1, d, rng.choice([d, d, 64]),
                     rng.choice(["bf16", "bf16", "f32"]), normalized=rng.random() < 0.3)
    B, H = _log_int(rng, 1, 8), rng.choice([4, 8, 12, 16, 32])
    if op == "hla3":
        dtype, d = rng.choice([("f32", 32), ("f32", 32), ("f32", 16), ("bf16", 64)])
        return _case(op, B, H, _log_int(rng, 64, 131072 // (B * H)), d, d, dtype)
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    d = rng.choice([64, 64, 128, 128, 32] if dtype == "bf16" else [16, 32, 64, 64, 128])
    most = 262144 if dtype == "bf16" else 65536
    if op == "backward":
        most //= 2
    if d == 128:
        most //= 2
    n = _log_int(rng, 32, most // (B * H))
    c = _case(op, B, H, n, d, d, dtype, normalized=rng.random() < 0.3)
    if op != "backward" and rng.random() < 0.4:  # a prefill, from nothing or from an earlier part of the prompt
        c["state_out"], c["state_in"] = True, rng.random() < 0.4
    if op == "forward" and not c["normalized"] and not c["state_out"] and rng.random() < 0.2:
        c["masked"] = False
    return c


def _tokens(c, seed, n, device, which):
    """q, k, v [B, H, n, d|dv] of the case's type; `which` tells the prompt's tokens from the call's."""
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) * 4 + which)
    B, H, d, dv = c["B"], c["H"], c["d"], c["dv"]

    def rows(width, unit):
        x = torch.randn((B, H, n, width), generator=g, device=device, dtype=torch.float32)
        if unit:
            x = x / x.norm(dim=-1, keepdim=True)
            x = x.abs() if c["normalized"] else x
        return x.to(DTYPES[c["dtype"]])

    return rows(d, True), rows(d, True), rows(dv, False)


def _prompt_parts(c, seed, device, dtype):
    """The parts of the case's state after a prompt of PROMPT tokens, from the defining sums."""
    q, k, v = (x.to(dtype) for x in _tokens(c, seed, PROMPT, device, 1))
    if c["op"] in ("ahla", "ahla_step"):
        A = (q @ k.mT).tril()
        return [k.mT @ v, k.sum(-2), k.mT @ (A @ v), k.mT @ A.sum(-1, keepdim=True)]
    if c["op"] == "step_sde":
        X = (q @ k.mT).tril() @ k
        return [k.mT @ k, X.mT @ v, X.sum(-2)]
    low = (k @ q.mT).tril(-1)  # the C and m before each token
    return [k.mT @ k, q.mT @ v, q.sum(-2), k.mT @ (low @ v), k.mT @ low.sum(-1, keepdim=True)]


def _pack(parts, B, H):
    return torch.cat([p.reshape(B, H, -1) for p in parts], dim=-1)


def _state_floats(c):
    f = hla.ahla_state_floats if c["op"] in ("ahla", "ahla_step") else (
        hla.hla2_sde_state_floats if c["op"] == "step_sde" else hla.hla2_state_floats)
    return f(c["d"], c["dv"])


def prepare(case, seed):
    c, dev = case, torch.device("cuda")
    B, H, n, d, dv, dt = c["B"], c["H"], c["n"], c["d"], c["dv"], DTYPES[c["dtype"]]
    s = {"case": c}
    q, k, v = _tokens(c, seed, n, dev, 0)
    if c["op"] in ("step", "step_sde", "ahla_step"):
        s["q"], s["k"], s["v"] = (x.reshape(B, H, -1) for x in (q, k, v))
        s["state"] = _pack(_prompt_parts(c, seed, dev, torch.float32), B, H).contiguous()
        s["out"] = torch.empty((B, H, dv), dtype=dt, device=dev)
        return s
    s["q"], s["k"], s["v"] = q, k, v
    if c["op"] == "backward":
        g = torch.Generator(device=dev)
        g.manual_seed(int(seed) * 4 + 2)
        s["dout"] = torch.randn((B, H, n, dv), generator=g, device=dev).to(dt)
        size = hla.hla2_backward_workspace_bytes(B, H, n, d, dv, 64, dt)
    else:
        s["out"] = torch.empty((B, H, n, dv), dtype=dt, device=dev)
        if c["state_in"]:
            s["state_in"] = _pack(_prompt_parts(c, seed, dev, torch.float32), B, H).contiguous()
        if c["state_out"]:
            s["state_out"] = torch.empty((B, H, _state_floats(c)), dtype=torch.float32, device=dev)
        size = {"forward": lambda: hla.hla2_workspace_bytes(B, H, n, d, dv, 128, dt),
                "ahla": lambda: hla.ahla_workspace_bytes(B, H, n, d, dv, 64, dt),
                "hla3": lambda: hla.hla3_workspace_bytes(B, H, n, d, dv, 32, dt)}[c["op"]]()
    s["workspace"] = hla.alloc_workspace(size, dev)
    return s


def run(s):
    c, norm = s["case"], s["case"]["normalized"]
    if c["op"] == "step":
        return hla.hla2_step(s["q"], s["k"], s["v"], s["state"], s["out"], normalized=norm, eps=EPS), s["state"]
    if c["op"] == "step_sde":
        return hla.hla2_step_sde(s["q"], s["k"], s["v"], s["state"], s["out"], normalized=norm, eps=EPS), s["state"]
    if c["op"] == "ahla_step":
        return hla.ahla_step(s["q"], s["k"], s["v"], s["state"], s["out"], normalized=norm, eps=EPS), s["state"]
    if c["op"] == "backward":
        return hla.hla2_backward(s["q"], s["k"], s["v"], s["dout"], normalized=norm, eps=EPS, workspace=s["workspace"])
    kept = {"state_in": s.get("state_in"), "state_out": s.get("state_out"), "workspace": s["workspace"]}
    if c["op"] == "ahla":
        out = hla.ahla_forward(s["q"], s["k"], s["v"], s["out"], normalized=norm, eps=EPS, **kept)
    elif c["op"] == "hla3":
        out = hla.hla3_forward(s["q"], s["k"], s["v"], s["out"], normalized=norm, eps=EPS, **kept)
    else:
        out = hla.hla2_forward(s["q"], s["k"], s["v"], s["out"], masked=c["masked"], normalized=norm, eps=EPS, **kept)
    return (out, s["state_out"]) if c["state_out"] else out


def work(case):
    c = case
    d, dv, size = c["d"], c["dv"], 2 if c["dtype"] == "bf16" else 4
    heads, tokens = c["B"] * c["H"], c["B"] * c["H"] * c["n"]
    state = 4 * heads * {"step": d * d + 2 * d * dv + 2 * d, "forward": d * d + 2 * d * dv + 2 * d,
                         "step_sde": d * d + d * dv + d}.get(c["op"], 2 * d * dv + 2 * d)
    io = tokens * size * (2 * d + 2 * dv)
    if c["op"] in ("step", "step_sde", "ahla_step"):
        return {"bytes": io + 2 * state, "flops": 3 * state / 4 * 2}
    C = TILE
    two = 2 * C * (d + dv) + C * C / 3 + 3 * d * d + 6 * d * dv + 2 * d * d * dv / C  # masked second order, a token
    if c["op"] == "backward":
        return {"bytes": tokens * size * (4 * d + 3 * dv), "flops": tokens * (
            two + 2 * (C * (dv + 3.5 * d) + 4 * d * dv + 4 * d * d + 2 * d * d * dv / C))}
    if c["op"] == "ahla":
        flops = tokens * 2 * (C * d / 2 + C * dv + 4 * d * dv + d * d * dv / C)
    elif c["op"] == "hla3":
        flops = tokens * 2 * (1.5 * C * d + 2 * C * dv + 4 * d * d + C * C / 6 + 5 * d * dv)
    else:
        flops = tokens * two
    return {"bytes": io + state * (c["state_in"] + c["state_out"]), "flops": flops}


def _out(num, den, c):
    return num / (den + EPS).unsqueeze(-1) if c["normalized"] else num


def _tiles(n):
    return [slice(t, min(n, t + TILE)) for t in range(0, n, TILE)]


def _forward64(q, k, v, c, parts=None):
    """(num, den) of second order, and the state tuple after the last token, tile by tile."""
    B, H, n, d = q.shape
    if parts is None:
        z = lambda *s: torch.zeros((B, H) + s, dtype=q.dtype, device=q.device)  # noqa: E731
        parts = [z(d, d), z(d, v.shape[-1]), z(d), z(d, v.shape[-1]), z(d, 1)]
    S, C, m, G, h = parts
    m, h = m.reshape(B, H, d, 1), h.reshape(B, H, d, 1)
    D, e = S @ C - G, S @ m - h
    nums, dens = [], []
    for t in _tiles(n):
        Q, K, V = q[:, :, t], k[:, :, t], v[:, :, t]
        X = (Q @ K.mT).tril() @ K + Q @ S
        if c["masked"]:
            T = (Q @ X.mT).tril()
            nums.append(T @ V + Q @ D)
            dens.append(T.sum(-1) + (Q @ e).squeeze(-1))
        else:
            T = (X @ Q.mT).tril()
            nums.append(T @ V + X @ C)
            dens.append(T.sum(-1) + (X @ m).squeeze(-1))
        D, e = D + X.mT @ V, e + X.sum(-2).unsqueeze(-1)
        S, C, m = S + K.mT @ K, C + Q.mT @ V, m + Q.sum(-2).unsqueeze(-1)
    keep = 1.0 if c["masked"] else 0.0
    return torch.cat(nums, -2), torch.cat(dens, -1), [S, C, m, keep * (S @ C - D), keep * (S @ m - e)]


def _ahla64(q, k, v, parts=None):
    B, H, n, d = q.shape
    v1 = torch.cat([v, torch.ones_like(v[..., :1])], -1)
    if parts is None:
        P = torch.zeros((B, H, d, v1.shape[-1]), dtype=q.dtype, device=q.device)
        E = P.clone()
    else:
        P, E = (torch.cat([parts[i], parts[i + 1].reshape(B, H, d, 1)], -1) for i in (0, 2))
    outs = []
    for t in _tiles(n):
        Q, K, V = q[:, :, t], k[:, :, t], v1[:, :, t]
        A = (Q @ K.mT).tril()
        R = A @ V + Q @ P
        outs.append(A @ R + Q @ E)
        P, E = P + K.mT @ V, E + K.mT @ R
    o = torch.cat(outs, -2)
    return o[..., :-1], o[..., -1], [P[..., :-1], P[..., -1], E[..., :-1], E[..., -1]]


def _third64(q, k, v):
    """Masked third order, tile by tile: with a_s = q_s.k_s, the state that the outputs read,
    num_t = q_t^T F_t, gains (k_s a_s) (q_s^T P_s) + k_s (k_s^T SQ_{s-1} k_s) v_s^T + (SK_{s-1} q_s) a_s v_s^T
    with every token."""
    B, H, n, d = q.shape
    z = lambda *s: torch.zeros((B, H) + s, dtype=q.dtype, device=q.device)  # noqa: E731
    SK, SQ, P, F = z(d, d), z(d, d), z(d, v.shape[-1]), z(d, v.shape[-1])
    outs = []
    for t in _tiles(n):
        Q, K, V = q[:, :, t], k[:, :, t], v[:, :, t]
        A = Q @ K.mT
        a = A.diagonal(dim1=-2, dim2=-1).unsqueeze(-1)
        low = A.tril()
        Y = Q @ P + low @ V
        b = ((K @ SQ) * K).sum(-1, keepdim=True) + A.triu(1).square().sum(-2).unsqueeze(-1)
        Z = a * Y + b * V
        U = Q @ SK + A.tril(-1) @ K  # rows SK_{s-1} q_s
        outs.append(Q @ F + low @ Z + (Q @ U.mT).tril() @ (a * V))
        F = F + K.mT @ Z + U.mT @ (a * V)
        SK, SQ, P = SK + K.mT @ K, SQ + Q.mT @ Q, P + K.mT @ V
    return torch.cat(outs, -2)


def exact(case, seed):
    c, dev = case, torch.device("cuda" if torch.cuda.is_available() else "cpu")
    B, H = c["B"], c["H"]
    q, k, v = (x.double() for x in _tokens(c, seed, c["n"], dev, 0))
    if c["op"] in ("step", "step_sde", "ahla_step"):
        st = [p.double() for p in _prompt_parts(c, seed, dev, torch.float32)]
        if c["op"] == "step_sde":
            S, D, e = st[0] + k.mT @ k, st[1], st[2].unsqueeze(-1)
            x = S @ q.mT
            D, e = D + x @ v, e + x
            return _out(q @ D, (q @ e).squeeze(-1), c).squeeze(-2), _pack([S, D, e], B, H)
        num, den, parts = _ahla64(q, k, v, st) if c["op"] == "ahla_step" else _forward64(q, k, v, c, st)
        return _out(num, den, c).squeeze(-2), _pack(parts, B, H)
    if c["op"] == "hla3":
        return _third64(q, k, v)
    if c["op"] == "backward":
        g = torch.Generator(device=dev)
        g.manual_seed(int(seed) * 4 + 2)
        dout = torch.randn((B, H, c["n"], c["dv"]), generator=g, device=dev).to(DTYPES[c["dtype"]]).double()
        leaves = [x.requires_grad_() for x in (q, k, v)]
        num, den, _ = _forward64(*leaves, c)
        return tuple(torch.autograd.grad(_out(num, den, c), leaves, dout))
    st = [p.double() for p in _prompt_parts(c, seed, dev, torch.float32)] if c["state_in"] else None
    num, den, parts = _ahla64(q, k, v, st) if c["op"] == "ahla" else _forward64(q, k, v, c, st)
    out = _out(num, den, c)
    return (out, _pack(parts, B, H)) if c["state_out"] else out

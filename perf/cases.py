"""Timed cases of the linear-attention layer: what a program that serves a model with it calls, through the public
binding (`paper_2406_07368_b200.binding.Context`).

Three kinds of pass:

  prefill   `la_prefill`, or `la_prefill_grouped` where the case has a group size: a prompt of T tokens per sequence,
            from an empty state or (cont) continuing from the state of the tokens before it
  decode    `la_decode_step`: one token for every sequence of the batch
  round     one speculative round: `la_verify_tree` on a draft tree per sequence, `la_accept_greedy` on the verifier's
            tokens, `la_commit` of the accepted path

A case says the kind and B (sequences), H (heads), d (head dimension), W (live taps of the convolution), io ("bf16" or
"f32"), phi ("elu1" or "relu"); prefill adds T, cont and group (0: exact layer), round adds N (nodes of the draft tree).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2406_07368_b200 import binding, workloads

MAX_DEPTH = 5          # depth of the draft trees, as in the repository's tree workloads


def _prefill(name, B, T, W=3, H=32, d=128, io="bf16", phi="elu1", cont=False, group=0):
    return {"name": name, "kind": "prefill", "B": B, "H": H, "d": d, "W": W, "io": io, "phi": phi, "T": T,
            "cont": cont, "group": group}


def _decode(name, B, W=3, H=32, d=128, io="bf16", phi="elu1"):
    return {"name": name, "kind": "decode", "B": B, "H": H, "d": d, "W": W, "io": io, "phi": phi}


def _round(name, B, N, W=3, H=32, d=128, io="bf16", phi="elu1"):
    return {"name": name, "kind": "round", "B": B, "H": H, "d": d, "W": W, "io": io, "phi": phi, "N": N}


def listed():
    return [
        # A single user's token: the inner step of interactive generation, 32 heads of one sequence.
        _decode("decode_one", B=1),
        # The decode step of a serving batch (the batched_decode shapes).
        _decode("decode_batch", B=64),
        # A chat turn: the short prompt of the prompt_gen shapes.
        _prefill("prompt_short", B=1, T=60),
        # A prompt of one user, longer and ragged (prompt_gen), that continues an earlier part of the conversation.
        _prefill("prompt_one", B=1, T=1700, cont=True),
        # The headline prefill: a batch of prompts (the llama7b_prefill shapes).
        _prefill("prefill_batch", B=4, T=2048),
        # A long document, ReLU features, five taps (the long_prefill shapes).
        _prefill("prefill_long", B=1, T=32768, W=5, phi="relu"),
        # The long convolution window (the prefill_taps32 shapes): a kernel of 63 under the causal mask.
        _prefill("prefill_taps32", B=4, T=2048, W=32),
        # The three-branch block as the paper trains it, groups of 64 (the grouped_block shapes).
        _prefill("prefill_grouped", B=4, T=2048, group=64),
        # A small model in full precision: 12 heads of dimension 64, fp32 in and out, ragged prompts.
        _prefill("prefill_fp32", B=4, T=1000, H=12, d=64, io="f32"),
        # A speculative round for one user: the whole of its latency is launches.
        _round("round_one", B=1, N=64),
        # The speculative round of a batch (the tree_verify shapes).
        _round("round_batch", B=16, N=64),
        # A round with smaller, ragged trees and a longer window (the taps of tree_verify_taps8).
        _round("round_taps8", B=7, N=29, W=8),
    ]


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi], odd ones as likely as even ones."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["prefill", "prefill", "grouped", "fp32", "decode", "round"])
    phi = rng.choice(["elu1", "elu1", "relu"])
    H = rng.choice([8, 12, 16, 32])
    if kind in ("prefill", "grouped"):
        T = _log(rng, 17, 16384)
        B = _log(rng, 1, max(1, min(16, 8 * 32768 // (H * T))))          # at most a quarter of the longest listed prompt
        if kind == "grouped":
            c = _prefill("", B, T, W=3, H=H, phi=phi, group=rng.choice([32, 64, 128]))
        else:
            c = _prefill("", B, T, W=rng.choice([1, 2, 3, 3, 4, 5, 8, 16, 32]), H=H, phi=phi, cont=rng.random() < 0.3)
    elif kind == "fp32":                                                 # what the fp32 case stands for: full precision
        T = _log(rng, 17, 1000)                                          # in either head dimension, and bf16 with d = 64
        io, d = rng.choice([("f32", 64), ("f32", 64), ("bf16", 64), ("f32", 128)])
        H = rng.choice([2, 8, 12])
        c = _prefill("", _log(rng, 1, max(1, 48 // H)), T, W=rng.choice([1, 3, 4]), H=H, d=d, io=io, phi=phi,
                     cont=rng.random() < 0.3)
    elif kind == "decode":
        io, d = rng.choice([("bf16", 128), ("bf16", 128), ("bf16", 64), ("f32", 64), ("f32", 128)])
        c = _decode("", _log(rng, 1, 128), W=rng.choice([1, 3, 3, 4, 8, 32]), H=H, d=d, io=io, phi=phi)
    else:
        c = _round("", _log(rng, 1, 32), rng.randint(5, 64), W=rng.choice([1, 3, 3, 4, 8, 16]), H=H, phi=phi)
    del c["name"]
    return c


# ---- inputs -------------------------------------------------------------------------------------------------------

def _normal(gen, shape, scale, dtype):
    x = torch.empty(shape, dtype=torch.float32, device="cuda").normal_(0.0, scale, generator=gen)
    return x.to(dtype)


def _phi(x, phi):
    x = x.float()
    return torch.relu(x) if phi == "relu" else torch.where(x > 0, x + 1.0, torch.exp(x))


def _state_after_prompt(ctx, case, gen, scale, tokens=256):
    """The running state of every sequence after a prompt of `tokens` tokens (formed sequence by sequence)."""
    st = ctx.new_state(case["B"])
    for b in range(case["B"]):
        k, v = (_normal(gen, (case["H"], tokens, case["d"]), scale, ctx.dtype) for _ in range(2))
        fk = _phi(k, case["phi"])
        st.S[b] = fk.transpose(1, 2) @ v.float()
        st.z[b] = fk.sum(1)
        if case["W"] > 1:
            st.win[b] = v[:, tokens - (case["W"] - 1):]
    st.pos.fill_(tokens)
    return st


def _trees(seed, B, N):
    """Draft trees, the drafted tokens, and the verifier's tokens such that one random path prefix of every tree is
    accepted (a uniform leaf, a uniform number of its path's nodes) and nothing else matches."""
    parent, accept = workloads.tree_batch(seed, 0, B, N, MAX_DEPTH)
    g = np.random.default_rng(seed)
    draft = g.permuted(np.arange(B * N, dtype=np.int32) + 1000).reshape(B, N)         # all different
    pred_root = g.integers(0, 1000, B, dtype=np.int32)                                # below 1000: matches no draft token
    pred = g.integers(0, 1000, (B, N), dtype=np.int32)
    for b in range(B):
        n = int(accept[b])
        while n >= 0:
            p = int(parent[b, n])
            if p < 0:
                pred_root[b] = draft[b, n]
            else:
                pred[b, p] = draft[b, n]
            n = p
    return parent, draft, pred_root, pred


def prepare(case, seed):
    B, H, d, W, kind = case["B"], case["H"], case["d"], case["W"], case["kind"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ctx = binding.Context(H, d, W, case["phi"], 1e-6 if case["phi"] == "relu" else 0.0, case["io"], max_depth=MAX_DEPTH)
    s = {"kind": kind, "ctx": ctx, "conv_w": _normal(gen, (H, d, W), W ** -0.5, torch.float32)}
    scale = d ** -0.5 if kind == "prefill" else 1.0
    tokens = {"prefill": (case.get("T"),), "decode": (), "round": (case.get("N"),)}[kind]
    s["q"], s["k"], s["v"] = (_normal(gen, (B, H, *tokens, d), scale, ctx.dtype) for _ in range(3))
    if kind == "prefill":
        s["group"], s["cont"] = case["group"], case["cont"]
        s["state"] = _state_after_prompt(ctx, case, gen, scale) if case["cont"] else ctx.new_state(B)
        need = ctx.la_prefill_workspace_bytes(B, case["T"])
        if need:                                            # a server lends its context the workspace it asks for
            ctx.la_set_workspace(torch.empty(need, dtype=torch.uint8, device="cuda"))
    else:
        s["state"] = _state_after_prompt(ctx, case, gen, scale)
    if kind == "round":
        names = ("parent", "draft", "pred_root", "pred")
        s.update({n: torch.from_numpy(x).cuda() for n, x in zip(names, _trees(seed, B, case["N"]))})
    return s


# ---- one pass -----------------------------------------------------------------------------------------------------

def run(s):
    ctx, st = s["ctx"], s["state"]
    if s["kind"] == "decode":
        out = {"o": ctx.la_decode_step(s["q"], s["k"], s["v"], s["conv_w"], st)}
    elif s["kind"] == "prefill":
        if s["group"]:
            o = ctx.la_prefill_grouped(s["q"], s["k"], s["v"], s["conv_w"], st, s["group"], 1.0, ctx.d ** -0.5)
        else:
            o = ctx.la_prefill(s["q"], s["k"], s["v"], s["conv_w"], st, init_state=s["cont"])
        out = {"o": o}
    else:
        o = ctx.la_verify_tree(s["q"], s["k"], s["v"], s["parent"], s["conv_w"], st)
        node, length, token = ctx.la_accept_greedy(s["parent"], s["draft"], s["pred_root"], s["pred"])
        path, committed = ctx.la_commit(s["k"], s["v"], s["parent"], node, st)
        out = {"o": o, "node": node, "length": length, "token": token, "path": path, "committed": committed}
    out.update(S=st.S, z=st.z, win=st.win, pos=st.pos)
    return out


# ---- what a pass cannot do without ----------------------------------------------------------------------------------

def work(case):
    B, H, d, W, kind = case["B"], case["H"], case["d"], case["W"], case["kind"]
    e = 2 if case["io"] == "bf16" else 4
    units = B * H
    state = (d * d + d) * 4 + (W - 1) * d * e                # S, z and the window of one (sequence, head)
    taps = H * d * W * 4
    if kind == "prefill":
        T, G = case["T"], case["group"]
        # q, k, v in and o out; the state out, and in where the prompt continues one.  Per token: the state update and
        # the readout (2 d^2 each), the taps; in the three-branch block also softmax attention to (G + 1) / 2 tokens.
        per_token = 4 * d * d + 2 * W * d + (4 * d * (G + 1) // 2 if G else 0)
        return {"bytes": units * (4 * T * d * e + state * (2 if case["cont"] else 1)) + taps, "flops": units * T * per_token}
    if kind == "decode":
        return {"bytes": units * (4 * d * e + 2 * state) + taps, "flops": units * (4 * d * d + 2 * W * d)}
    # A round: q, k, v, o of the nodes, the state in and out, and the trees with their tokens.  Per node: the readout of
    # the state, its ancestors (at most MAX_DEPTH), the taps; then the rank-1 updates of the accepted path.
    N = case["N"]
    flops = units * (N * (2 * d * d + 4 * d * MAX_DEPTH + 2 * W * d) + 2 * d * d * MAX_DEPTH // 2)
    return {"bytes": units * (4 * N * d * e + 2 * state) + taps + B * N * 12, "flops": flops}


def tolerance(case):
    # bf16: phi, the scores and the copy of the state that the products read are rounded to bf16 (2^-9 each), and so is
    # the output; fp32: sums of up to a few thousand fp32 products.  Whole numbers (paths, lengths, tokens) are exact.
    return {"rel": 1e-2} if case["io"] == "bf16" else {"rel": 1e-5}

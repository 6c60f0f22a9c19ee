"""The measured workloads of the linear-attention library, called the way a program calls them.

A case is one attention layer's call on tensors that are already on the GPU, through ``paper_2510_08318_b200.linattn.LinAttn``:

  op       "forward"      linattn_forward (inference; the operator itself)
           "mixed"        linattn_forward_mixed (Eq. 8, while softmax attention is being transferred)
           "backward"     linattn_backward (recomputes S and z)
           "train"        forward, then the backward that takes S and z over from it (LINATTN_OPT_REUSE_STATE)
           "train_mixed"  forward_mixed, then backward_mixed with the softmax branch's gradient
  dtype    storage of q, k, v and the outputs; weights: type in which W_q, W_k are given (fp32 master weights or bf16)
  layout   0 = [B][H][n][d], 1 = [B][n][H][d] (the order a DiT's projections leave)
  per_head 1 = every head has its own W_q, W_k, 0 = one shared matrix
  relu     the ReLU kernel function instead of the Hedgehog feature map
  tails    5 % of the keys' entries drawn from a Student-t with 3 degrees of freedom

Shapes are those of the repository's own workloads (Wan-1.3B and -14B layers at 480p and 720p, the CogVideoX-2B-shaped
layer of head dimension 64, the tiny fp32 case) and smaller or ragged ones of the same kind.
"""
from __future__ import annotations

import math

import torch

_DT = {"f32": torch.float32, "bf16": torch.bfloat16}


def _case(name, op, B, H, n, d, dtype, weights, layout=0, per_head=1, relu=0, tails=0, r=0.0):
    c = {"op": op, "B": B, "H": H, "n": n, "d": d, "dtype": dtype, "weights": weights, "layout": layout,
         "per_head": per_head, "relu": relu, "tails": tails, "r": r}
    if name:
        c = {"name": name, **c}
    return c


def listed():
    return [
        # the smallest call: the tiny fp32 correctness shape; launches and latency
        _case("fwd_tiny_f32", "forward", 1, 2, 1024, 64, "f32", "f32"),
        # one latent frame of 30 x 52 tokens through a Wan-1.3B layer: latency of the bf16 path
        _case("fwd_one_frame", "forward", 1, 12, 1560, 128, "bf16", "bf16"),
        # the headline workload: Wan-1.3B layer, 81 frames at 480p
        _case("fwd_480p", "forward", 1, 12, 32760, 128, "bf16", "bf16"),
        # the longest sequence: Wan-14B layer at 720p
        _case("fwd_720p", "forward", 1, 40, 75600, 128, "bf16", "bf16"),
        # head dimension 64: CogVideoX-2B-shaped joint text + video sequence, odd tail
        _case("fwd_d64_joint", "forward", 1, 30, 17776, 64, "bf16", "bf16"),
        # transfer from softmax attention as a training loop runs it forward: CFG pair, token-major, fp32 master weights
        _case("mixed_pair_fp32w", "mixed", 2, 12, 16390, 128, "bf16", "f32", layout=1, r=0.5),
        # full-precision inference (numerics reference of a deployment) at the headline shape
        _case("fwd_f32_480p", "forward", 1, 12, 32760, 128, "f32", "f32"),
        # gradients of the headline layer
        _case("bwd_480p", "backward", 1, 12, 32760, 128, "bf16", "bf16"),
        # training step of a Wan-14B layer with Eq. 8 and heavy-tailed keys: the largest training call
        _case("train_14b_mixed", "train_mixed", 1, 40, 32760, 128, "bf16", "bf16", tails=1, r=0.7),
        # training step of the head-dimension-64 layer
        _case("train_d64_joint", "train", 1, 30, 17776, 64, "bf16", "bf16"),
        # training with fp32 master weights and bf16 activations, token-major, shorter clip
        _case("train_fp32w", "train", 1, 12, 14040, 128, "bf16", "f32", layout=1),
        # a small fp32 training step of odd length with one shared feature map (gradient checks, toy models)
        _case("train_small_f32", "train", 2, 3, 777, 64, "f32", "f32", per_head=0),
    ]


#: elements (B * H * n * d) of the largest listed case of each kind: a drawn case costs no more
_MOST = {"forward": 40 * 75600 * 128, "mixed": 40 * 32760 * 128, "slow": 12 * 14040 * 128, "grad": 40 * 32760 * 128}


def draw(rng):
    op = rng.choices(["forward", "mixed", "backward", "train", "train_mixed"], [6, 2, 2, 3, 1])[0]
    d = rng.choices([64, 128], [2, 3])[0]
    dtype = rng.choices(["bf16", "f32"], [4, 1])[0]
    weights = "f32" if dtype == "f32" else rng.choices(["bf16", "f32"], [3, 1])[0]
    relu = 1 if rng.random() < 0.08 else 0
    B = rng.choice([1, 1, 2])
    H = rng.choice([2, 3, 12, 12, 16, 30, 40])
    n = int(round(math.exp(rng.uniform(math.log(190.0), math.log(75600.0)))))
    grad = op in ("backward", "train", "train_mixed")
    if dtype == "f32" or (grad and (d == 64 or weights == "f32" or relu)):
        most = _MOST["slow"]
    else:
        most = _MOST["grad" if grad else op]
    n = max(64, min(n, most // (B * H * d)))
    return _case(None, op, B, H, n, d, dtype, weights, layout=rng.choice([0, 1]), per_head=rng.choice([1, 1, 0]), relu=relu,
                 tails=rng.choices([0, 1], [3, 1])[0], r=round(rng.uniform(0.05, 0.95), 2) if "mixed" in op else 0.0)


def _inputs(case, seed):
    """q, k, v (and dout, the softmax branch's output a) in the case's layout and type, Wq, Wk; the same scales as the
    repository's synthetic workloads: q, k, v ~ N(0, 1/d) (N(0, 1) in fp32), logits of unit variance."""
    B, H, n, d = case["B"], case["H"], case["n"], case["d"]
    dt = _DT[case["dtype"]]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    sigma = 1.0 if case["dtype"] == "f32" else 1.0 / math.sqrt(d)
    shape = (B, n, H, d) if case["layout"] else (B, H, n, d)

    def normal(*s):
        return torch.randn(*s, generator=gen, device="cuda", dtype=torch.float32)

    x = {}
    for name in ("q", "k", "v"):
        t = normal(*shape).mul_(sigma)
        if name == "k" and case["tails"]:
            chi = (normal(*shape).square_() + normal(*shape).square_() + normal(*shape).square_()).div_(3.0)
            tail = normal(*shape).mul_(sigma).div_(chi.sqrt_())
            t = torch.where(torch.rand(*shape, generator=gen, device="cuda") < 0.05, tail, t)
        x[name] = t.to(dt)
    wshape = (H, d, d // 2) if case["per_head"] else (d, d // 2)
    for name in ("Wq", "Wk"):
        x[name] = normal(*wshape).div_(math.sqrt(d) * sigma).to(_DT[case["weights"]])
    if "mixed" in case["op"]:
        x["a"] = normal(*shape).mul_(sigma / math.sqrt(n)).to(dt)   # an average of about n values
    if case["op"] not in ("forward", "mixed"):
        x["dout"] = normal(*shape).mul_(sigma).to(dt)
    return x


def prepare(case, seed):
    """The layer's context with its weights set, and the activations on the GPU."""
    from paper_2510_08318_b200 import linattn

    x = _inputs(case, seed)
    ctx = linattn.LinAttn(case["H"], case["d"], max_B=case["B"], max_n=case["n"])
    ctx.set_option(linattn.OPT_LAYOUT, case["layout"])
    ctx.set_option(linattn.OPT_KERNEL_FUNCTION, case["relu"])
    if case["op"].startswith("train"):
        ctx.set_option(linattn.OPT_REUSE_STATE, 1)   # the forward -> backward order of a training step
    if not case["relu"]:
        ctx.set_feature_map(x["Wq"], x["Wk"])
    for name in ("q", "k", "v", "a", "dout"):
        if name in x and case["layout"]:
            # LinAttn reads B, H, n, d from the shape: the token-major memory is passed under the [B, H, n, d] shape
            x[name] = x[name].view(case["B"], case["H"], case["n"], case["d"])
    return {"case": dict(case), "ctx": ctx, **x}


def run(state):
    c, ctx = state["case"], state["ctx"]
    q, k, v = state["q"], state["k"], state["v"]
    out = {}
    if c["op"] in ("forward", "train"):
        out["out"] = ctx.forward(q, k, v)
    elif c["op"] in ("mixed", "train_mixed"):
        out["out"] = ctx.forward_mixed(q, k, v, state["a"], c["r"])
    if c["op"] in ("backward", "train"):
        g = ctx.backward(q, k, v, state["dout"], per_head=bool(c["per_head"]))
        names = ("dq", "dk", "dv", "dWq", "dWk")
    elif c["op"] == "train_mixed":
        g = ctx.backward_mixed(q, k, v, state["a"], c["r"], state["dout"], per_head=bool(c["per_head"]))
        names = ("dq", "dk", "dv", "dWq", "dWk", "da", "dr")
    else:
        return out
    for name, t in zip(names, g):
        if not (c["relu"] and name in ("dWq", "dWk")):   # the ReLU kernel function has no weights
            out[name] = t
    return out


def work(case):
    """Every input read once, every output written once; the contractions of Eq. 5 and Eq. 6 and of their gradients."""
    B, H, n, d = case["B"], case["H"], case["n"], case["d"]
    e = 2 if case["dtype"] == "bf16" else 4
    we = 2 if case["weights"] == "bf16" else 4
    T = B * H * n
    mats = (H if case["per_head"] else 1) * d * (d // 2)
    mixed, op = "mixed" in case["op"], case["op"]
    tensors, flops = 0, 0
    logits = 0 if case["relu"] else d * d          # x W of one token (2 * d * d/2)
    if op in ("forward", "mixed", "train", "train_mixed"):
        tensors += 4 + mixed                       # q, k, v (, a) in, out written
        flops += 2 * logits + 4 * d * d            # both feature maps, S += phi(k)^T v, phi(q) S
    if op in ("backward", "train", "train_mixed"):
        if op == "backward":
            tensors += 3                           # q, k, v in
            flops += 2 * logits + 2 * d * d        # both feature maps, S
        tensors += 4 + mixed                       # dout in, dq, dk, dv (, da) written
        flops += 4 * logits + 8 * d * d            # dx = du W^T and dW on both sides; dO S^T, dS, V dS^T, phi dS
    wbytes = 0 if case["relu"] else 2 * mats * we + (2 * mats * 4 if op not in ("forward", "mixed") else 0)
    return {"bytes": float(tensors * T * d * e + wbytes), "flops": float(flops * T)}


def tolerance(case):
    # bf16: rounding of the outputs (1.7e-3) and of phi, phi / den, du where they are tensor-core operands (about 3e-3 in
    # all).  fp32: about 1e-6 against 64 bits (3e-6 for the gradients), two orders of summation.
    if case["dtype"] == "bf16":
        return {"rel": 1e-2}
    return {"rel": 1e-5}


def exact(case, seed):
    """Eq. 5, Eq. 6, Eq. 8 and their gradients in 64 bits, head by head: the chain rule written out in plain torch."""
    B, H, n, d = case["B"], case["H"], case["n"], case["d"]
    x = _inputs(case, seed)
    op, relu, m = case["op"], case["relu"], d // 2
    r = min(max(case["r"], 0.0), 1.0)
    mixed, fwd, grad = "mixed" in op, op in ("forward", "mixed", "train", "train_mixed"), op in ("backward", "train", "train_mixed")

    def head(t, b, h):
        return (t[b, :, h] if case["layout"] else t[b, h]).double()

    def blank():
        return torch.empty(x["q"].shape, dtype=torch.float64, device="cuda")

    def put(t, b, h, val):
        if case["layout"]:
            t[b, :, h] = val
        else:
            t[b, h] = val

    def phi(t, W):
        if relu:
            return t.clamp(min=0.0)
        u = t @ W
        return torch.cat([torch.softmax(u, -1), torch.softmax(-u, -1)], -1)

    def back(t, p, dp, W):
        """Gradients of phi's input and of W, given those of phi."""
        if relu:
            return dp * (t > 0), None
        pp, pn, gp, gn = p[:, :m], p[:, m:], dp[:, :m], dp[:, m:]
        du = pp * (gp - (pp * gp).sum(-1, keepdim=True)) - pn * (gn - (pn * gn).sum(-1, keepdim=True))
        return du @ W.t(), t.t() @ du

    res = {}
    if fwd:
        res["out"] = blank()
    if grad:
        for name in ("dq", "dk", "dv"):
            res[name] = blank()
        if not relu:
            for name in ("dWq", "dWk"):
                res[name] = torch.zeros((H, d, m) if case["per_head"] else (d, m), dtype=torch.float64, device="cuda")
        if mixed:
            res["da"] = r * x["dout"].double()
            dr = torch.zeros(1, dtype=torch.float64, device="cuda")
            res["dr"] = dr
    for b in range(B):
        for h in range(H):
            q, k, v = head(x["q"], b, h), head(x["k"], b, h), head(x["v"], b, h)
            Wq, Wk = ((x[w][h] if case["per_head"] else x[w]).double() for w in ("Wq", "Wk"))
            pq, pk = phi(q, Wq), phi(k, Wk)
            S, z = pk.t() @ v, pk.sum(0)
            den = (pq @ z)[:, None]
            o = (pq @ S) / den
            a = head(x["a"], b, h) if mixed else None
            if fwd:
                put(res["out"], b, h, r * a + (1.0 - r) * o if mixed else o)
            if not grad:
                continue
            go = head(x["dout"], b, h)
            if mixed:
                dr += (go * (a - o)).sum()
                go = (1.0 - r) * go
            dnum, dden = go / den, -(go * o).sum(-1, keepdim=True) / den
            dS, dz = pq.t() @ dnum, (pq * dden).sum(0)
            dq, dWq = back(q, pq, dnum @ S.t() + dden * z, Wq)
            dk, dWk = back(k, pk, v @ dS.t() + dz, Wk)
            put(res["dq"], b, h, dq)
            put(res["dk"], b, h, dk)
            put(res["dv"], b, h, pk @ dS)
            if not relu:
                for name, g in (("dWq", dWq), ("dWk", dWk)):
                    if case["per_head"]:
                        res[name][h] += g
                    else:
                        res[name] += g
    shape = (B, H, n, d)
    return {name: t.view(shape) if name in ("out", "dq", "dk", "dv", "da") else t for name, t in res.items()}

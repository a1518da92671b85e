"""What the performance of this package is measured on.

Each case is one pass through the package's public entry points
(``paper_2609_08443_gb300.binding``) at a size that real use of Sketch Attention
meets: serving one user, a batch of users, the training step at the widths and
prototype counts of the evaluation workloads, the stacked refinement (per-user
queries), the key projection, the token-wise comparison, fp32 inputs, and a
prototype count that is not a power of two.

A case is a dict of plain values:
  op      fwd       sketch and lse                       (sa_sketch_fwd)
          step      sketch, dK, dV, dQ                   (sa_sketch + autograd)
          per_user  the same with Q [B, H, P, d]         (sa_sketch + autograd)
          x         sketch, lse, dX, dQ, dWk             (sa_sketch_fwd_x, sa_sketch_bwd_x)
          tokenwise sketch, lse_tok, dK, dV, dQ          (sa_sketch_*_tokenwise)
  dtype   bf16 | f32          H, P, d   heads, prototypes, width per head
  users   B histories, log-uniform in [lo, hi] (lo = hi: all alike), drawn from
          len_seed; n_long more of L_long tokens, spread among them
  q_std   standard deviation of the prototypes

The host-memory step is not listed: it runs the same kernels as ``step`` behind
copies that the host link paces.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2609_08443_gb300 import binding


def _case(op, H, P, d, B, lo, hi, dtype="bf16", n_long=0, L_long=0, q_std=1.0, len_seed=1, name=None):
    c = dict(op=op, dtype=dtype, H=H, P=P, d=d, B=B, lo=lo, hi=hi, n_long=n_long, L_long=L_long, q_std=q_std,
             len_seed=len_seed)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # serving: one request, one user's history, the smallest call there is
        _case("fwd", 8, 256, 64, B=1, lo=1531, hi=1531, name="serve_1user"),
        # the 4096-token fp32 workload: a single user in full precision
        _case("fwd", 1, 64, 64, B=1, lo=4096, hi=4096, dtype="f32", name="fwd_f32_4096"),
        # serving or evaluation of a ragged batch of 32 users, H = 4, d = 64
        _case("fwd", 4, 256, 64, B=32, lo=1024, hi=16384, len_seed=2, name="fwd_batch32"),
        # training step at d = 64: 64 users with histories spread over 512 .. 100K tokens
        _case("step", 8, 256, 64, B=64, lo=512, hi=100000, len_seed=3, name="step_64users_d64"),
        # training step at d = 128, P = 512 on 100K-token histories, the flagship shape
        _case("step", 8, 512, 128, B=16, lo=100000, hi=100000, q_std=0.02, name="step_100k_d128"),
        # ragged extremes: one 1M-token history among a thousand of 1 .. 512 tokens
        _case("step", 8, 256, 64, B=1024, lo=1, hi=512, n_long=1, L_long=1048576, len_seed=5,
              name="step_extremes"),
        # a small fine-tuning batch at the flagship shape: launches and the last wave count
        _case("step", 8, 512, 128, B=4, lo=300, hi=3000, len_seed=6, name="step_small_d128"),
        # stacked refinement: every user brings their own queries
        _case("per_user", 8, 512, 128, B=12, lo=5000, hi=60000, len_seed=7, name="step_per_user_q"),
        # training step with the key projection, X as keys (through W_K) and values
        _case("x", 8, 512, 128, B=12, lo=5000, hi=60000, len_seed=8, name="step_key_projection"),
        # the token-wise normalisation the method is compared with
        _case("tokenwise", 8, 512, 128, B=12, lo=5000, hi=60000, len_seed=9, name="step_tokenwise"),
        # training step at 1024 prototypes (the method's final sketch length)
        _case("step", 8, 1024, 128, B=6, lo=5000, hi=60000, len_seed=10, name="step_p1024"),
        # fp32 training step, and a prototype count that is no power of two
        _case("step", 4, 200, 64, B=8, lo=200, hi=5000, dtype="f32", len_seed=11, name="step_f32_p200"),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["serve", "batch", "step64", "step128", "extremes", "per_user", "x", "tokenwise", "large_p",
                       "f32", "odd_p"])
    seed = rng.randrange(1 << 30)
    while True:
        if kind == "serve":
            n = logint(100, 100000)
            c = _case("fwd", rng.choice([4, 8]), rng.choice([128, 256, 512]), rng.choice([64, 128]), B=1, lo=n, hi=n)
        elif kind == "batch":
            c = _case("fwd", rng.choice([4, 8]), rng.choice([128, 256, 512]), rng.choice([64, 128]),
                      B=logint(2, 128), lo=logint(50, 1000), hi=logint(1000, 50000))
        elif kind == "step64":
            c = _case("step", rng.choice([4, 8]), rng.choice([128, 256, 512]), 64, B=logint(1, 64),
                      lo=logint(50, 1000), hi=logint(1000, 100000))
        elif kind == "step128":
            c = _case("step", rng.choice([4, 8]), rng.choice([128, 256, 512]), 128, B=logint(1, 32),
                      lo=logint(50, 5000), hi=logint(5000, 100000), q_std=rng.choice([0.02, 1.0]))
        elif kind == "extremes":
            c = _case("step", 8, 256, rng.choice([64, 128]), B=logint(100, 1000), lo=1, hi=logint(100, 512),
                      n_long=rng.randint(0, 1), L_long=logint(20000, 500000))
        elif kind == "per_user":
            c = _case("per_user", rng.choice([4, 8]), rng.choice([256, 512]), rng.choice([64, 128]),
                      B=logint(1, 24), lo=logint(100, 3000), hi=logint(3000, 60000))
        elif kind == "x":
            c = _case("x", rng.choice([4, 8]), rng.choice([256, 512]), rng.choice([64, 128]), B=logint(1, 24),
                      lo=logint(100, 3000), hi=logint(3000, 60000))
        elif kind == "tokenwise":
            c = _case("tokenwise", rng.choice([4, 8]), rng.choice([256, 512, 1024]), 128, B=logint(1, 24),
                      lo=logint(100, 3000), hi=logint(3000, 60000))
        elif kind == "large_p":
            c = _case("step", rng.choice([4, 8]), rng.choice([1024, 2048]), rng.choice([64, 128]), B=logint(1, 8),
                      lo=logint(100, 3000), hi=logint(3000, 60000))
        elif kind == "f32":
            c = _case("step", rng.choice([1, 4]), rng.randint(16, 256), rng.choice([32, 64, 128]),
                      B=logint(1, 12), lo=logint(20, 300), hi=logint(300, 5000), dtype="f32")
        else:
            c = _case("step", rng.choice([1, 4]), rng.randint(16, 400), rng.choice([32, 64, 96]), B=logint(1, 12),
                      lo=logint(20, 300), hi=logint(300, 5000))
        c["len_seed"] = seed
        # no drawn case costs more than the listed ones of its kind of arithmetic
        cap = 60e9 if kind in ("f32", "odd_p") else 4e12
        if work(c)["flops"] <= cap:
            return c


# ------------------------------------------------------------------ inputs

def _lengths(case):
    rng = random.Random(case["len_seed"])
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    lens = [min(case["hi"], max(case["lo"], int(round(math.exp(rng.uniform(lo, hi)))))) for _ in range(case["B"])]
    for _ in range(case["n_long"]):
        lens.insert(rng.randrange(len(lens) + 1), case["L_long"])
    return lens


def prepare(case, seed):
    """Inputs on the GPU: K, V (or X), packed offsets, prototypes, upstream gradient."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed * 7919 + 13)
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    H, P, d = case["H"], case["P"], case["d"]

    def normal(shape, std=1.0, dtype=dt):
        x = torch.empty(shape, dtype=dtype, device=dev)
        return x.normal_(0.0, std, generator=g)

    lens = _lengths(case)
    cu = [0]
    for n in lens:
        cu.append(cu[-1] + n)
    B, N = len(lens), cu[-1]
    s = dict(op=case["op"], lens=lens, cu=torch.tensor(cu, dtype=torch.int32, device=dev))
    s["K"] = normal((N, H, d))
    if case["op"] == "x":
        s["Wk"] = normal((H, d, d), 1.0 / math.sqrt(d))
    else:
        s["V"] = normal((N, H, d))
    s["Q"] = normal((B, H, P, d) if case["op"] == "per_user" else (H, P, d), case["q_std"])
    if case["op"] != "fwd":
        s["dsketch"] = normal((B, H, P, d), 1.0, torch.float32)
    if case["op"] in ("step", "per_user"):
        for k in ("K", "V", "Q"):
            s[k].requires_grad_(True)
    return s


def run(state):
    s = state
    op, K, cu, Q = s["op"], s["K"], s["cu"], s["Q"]
    if op == "fwd":
        sketch, lse = binding.sa_sketch_fwd(K, s["V"], cu, Q, want_lse=True)
        return {"sketch": sketch, "lse": lse}
    if op in ("step", "per_user"):
        sketch = binding.sa_sketch(K, s["V"], cu, Q)
        dK, dV, dQ = torch.autograd.grad(sketch, (K, s["V"], Q), s["dsketch"])
        return {"sketch": sketch.detach(), "dK": dK, "dV": dV, "dQ": dQ}
    if op == "x":
        sketch, lse = binding.sa_sketch_fwd_x(K, cu, Q, s["Wk"], want_lse=True)
        dX, dQ, dWk = binding.sa_sketch_bwd_x(K, cu, Q, s["Wk"], s["dsketch"], lse=lse)
        return {"sketch": sketch, "lse": lse, "dX": dX, "dQ": dQ, "dWk": dWk}
    sketch, lse = binding.sa_sketch_fwd_tokenwise(K, s["V"], cu, Q, want_lse=True)
    dK, dV, dQ = binding.sa_sketch_bwd_tokenwise(K, s["V"], cu, Q, s["dsketch"], sketch=sketch, lse=lse)
    return {"sketch": sketch, "lse": lse, "dK": dK, "dV": dV, "dQ": dQ}


def work(case):
    """Each input read once, each output written once; two contractions of P x d
    per token and head forward (scores, sketch) and four backward (dV, dA, dK, dQ)."""
    lens = _lengths(case)
    B, N = len(lens), sum(lens)
    H, P, d, op = case["H"], case["P"], case["d"], case["op"]
    eb = 2 if case["dtype"] == "bf16" else 4
    tok = N * H * d * eb                     # one per-token tensor
    sk = B * H * P * d * 4                   # sketch or its gradient
    q = H * P * d * (B if op == "per_user" else 1)
    nbytes = sk + q * eb + (B + 1) * 4
    nbytes += tok * (1 if op == "x" else 2)
    flops = 4 * P * d * N * H
    if op in ("fwd", "x"):
        nbytes += N * H * 4                  # lse
    if op == "tokenwise":
        nbytes += B * H * P * 4
    if op != "fwd":
        flops += 8 * P * d * N * H
        nbytes += sk + tok * (1 if op == "x" else 2)
        nbytes += q * (eb if op in ("step", "per_user") else 4)
    if op == "x":
        nbytes += H * d * d * (eb + 4)
        flops += 6 * H * P * d * d
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------ 64-bit values

def exact(case, seed):
    """The same outputs in float64, user by user, in plain torch."""
    if work(case)["flops"] > 2.5e12:
        return None
    s = prepare(case, seed)
    f64 = torch.float64
    op, lens = s["op"], s["lens"]
    K, Q = s["K"].detach(), s["Q"].detach()
    V = K if op == "x" else s["V"].detach()
    N, H, d = K.shape
    P = Q.shape[-2]
    B = len(lens)
    dev = K.device
    scale = 1.0 / math.sqrt(d)
    step = op != "fwd"
    Wk = s["Wk"].to(f64) if op == "x" else None
    sketch = torch.zeros((B, H, P, d), dtype=f64, device=dev)
    lse_shape = (B, H, P) if op == "tokenwise" else (N, H)
    lse = torch.zeros(lse_shape, dtype=f64, device=dev)
    if step:
        dK = torch.zeros((N, H, d), dtype=f64, device=dev)
        dV = torch.zeros((N, H, d), dtype=f64, device=dev)
        dQ = torch.zeros(tuple(Q.shape), dtype=f64, device=dev)
        dWk = torch.zeros((H, d, d), dtype=f64, device=dev)
    t0 = 0
    chunk = 16384
    for b, n in enumerate(lens):
        q = (Q[b] if op == "per_user" else Q).to(f64)                       # H P d
        G = s["dsketch"][b].to(f64) if step else None
        parts = [(t, min(t + chunk, t0 + n)) for t in range(t0, t0 + n, chunk)]

        def load(a, e):
            x = K[a:e].to(f64).transpose(0, 1)                              # H t d
            v = x if op == "x" else V[a:e].to(f64).transpose(0, 1)
            k = torch.bmm(x, Wk) if op == "x" else x
            return x, k, v

        if op == "tokenwise":  # normalised over the user's tokens, per prototype
            m = torch.full((H, 1, P), -math.inf, dtype=f64, device=dev)
            z = torch.zeros((H, 1, P), dtype=f64, device=dev)
            for a, e in parts:
                _, k, _ = load(a, e)
                S = torch.bmm(k, q.transpose(1, 2)) * scale
                m2 = torch.maximum(m, S.amax(1, keepdim=True))
                z = z * torch.exp(m - m2) + torch.exp(S - m2).sum(1, keepdim=True)
                m = m2
            L = m + torch.log(z)                                            # H 1 P
            lse[b] = L[:, 0]
        for a, e in parts:
            x, k, v = load(a, e)
            S = torch.bmm(k, q.transpose(1, 2)) * scale                     # H t P
            if op != "tokenwise":
                L = torch.logsumexp(S, 2, keepdim=True)
                lse[a:e] = L[:, :, 0].transpose(0, 1)
            A = torch.exp(S - L)
            sketch[b] += torch.bmm(A.transpose(1, 2), v)
            if step and op != "tokenwise":
                dv = torch.bmm(A, G)
                dA = torch.bmm(v, G.transpose(1, 2))
                dS = A * (dA - (A * dA).sum(2, keepdim=True)) * scale
                dk = torch.bmm(dS, q)
                dq = torch.bmm(dS.transpose(1, 2), k)
                if op == "x":
                    dWk += torch.bmm(x.transpose(1, 2), dk)
                    dk = torch.bmm(dk, Wk.transpose(1, 2)) + dv
                dK[a:e] = dk.transpose(0, 1)
                dV[a:e] = dv.transpose(0, 1)
                if op == "per_user":
                    dQ[b] += dq
                else:
                    dQ += dq
        if op == "tokenwise":
            D = (G * sketch[b]).sum(2)[:, None, :]                          # H 1 P
            for a, e in parts:
                _, k, v = load(a, e)
                A = torch.exp(torch.bmm(k, q.transpose(1, 2)) * scale - L)
                dS = A * (torch.bmm(v, G.transpose(1, 2)) - D) * scale
                dV[a:e] = torch.bmm(A, G).transpose(0, 1)
                dK[a:e] = torch.bmm(dS, q).transpose(0, 1)
                dQ += torch.bmm(dS.transpose(1, 2), k)
        t0 += n
    if op == "fwd":
        return {"sketch": sketch, "lse": lse}
    if op == "x":
        return {"sketch": sketch, "lse": lse, "dX": dK, "dQ": dQ, "dWk": dWk}
    if op == "tokenwise":
        return {"sketch": sketch, "lse": lse, "dK": dK, "dV": dV, "dQ": dQ}
    return {"sketch": sketch, "dK": dK, "dV": dV, "dQ": dQ}

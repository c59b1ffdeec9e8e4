"""Performance cases of the library: what a program that uses it has it do, with sizes.

Every case is one pass of one attention layer (or of the projection gates behind it) through the
public entry points of ``paper_2604_00754_b200.binding`` and ``.host``, the way a model calls them:
a fresh permutation per layer and pass, then the forward, or the forward with saved state and the
backward.  Kinds:

  forward  SA alone, inference: make_perm + sa_forward
  gated    SA + SWA under the scalar gates, inference: make_perm + sa_swa_gated_forward
  rope     the same with rotary embedding by original positions: make_perm + sa_swa_gated_forward_rope
  train    forward that saves its state + backward (gated, or SA alone)
  gates    projection gates of both paths, forward + backward
  host     HostForward: tensors in pinned host memory, copies in and out included

``listed()`` names the shapes; ``draw()`` gives further shapes of the same kinds and ranges.
"""
import math

import torch

from paper_2604_00754_b200 import binding as sa
from paper_2604_00754_b200.host import HostForward

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _attn(name, kind, dtype, B, Hq, Hkv, n, d, w, causal=True, linear=False, layout="bhnd",
          gated=True):
    c = dict(kind=kind, dtype=dtype, B=B, Hq=Hq, Hkv=Hkv, n=n, d=d, w=w, causal=causal,
             linear=linear, layout=layout, gated=gated)
    if name:
        c["name"] = name
    return c


def _gates(name, dtype, rows, dm, dual):
    c = dict(kind="gates", dtype=dtype, rows=rows, dm=dm, dual=dual)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest configuration (one head, 256 tokens, fp32): a numerical check or a toy model,
        # where launches and host work are everything.
        _attn("tiny_f32_forward", "forward", "f32", 1, 1, 1, 256, 64, 32, gated=False),
        # A short prompt of ragged length through a layer of the 32/8-head shape: time to first token.
        _attn("short_prompt_gated", "gated", "bf16", 1, 32, 8, 700, 128, 256),
        # A single multi-head layer at ordinary size, SA alone (configuration 2).
        _attn("layer_4096_forward", "forward", "bf16", 2, 16, 16, 4096, 128, 256, gated=False),
        # Prefill of 32k tokens, 32/8 heads, both branches gated: the benchmark's step.
        _attn("prefill_32k_gated", "gated", "bf16", 1, 32, 8, 32768, 128, 1024),
        # One layer of the 131072-token prefill, 32/4 heads: the largest case.
        _attn("prefill_128k_gated", "gated", "bf16", 1, 32, 4, 131072, 128, 2048),
        # One layer of the pre-training step: 12 heads of 64, narrow window, forward + backward.
        _attn("pretrain_gated_train", "train", "bf16", 8, 12, 12, 4096, 64, 128),
        # The shape of the paper's efficiency table: SA alone, forward + backward, 16 heads of 64.
        _attn("table_2048_sa_train", "train", "bf16", 16, 16, 16, 2048, 64, 256, gated=False),
        # Retrofitting a 32/8-head model on documents of odd length; activations are token-major
        # ([B,n,H,d]), as a projection leaves them.
        _attn("finetune_10007_gated_train", "train", "bf16", 1, 32, 8, 10007, 128, 1024,
              layout="bnhd"),
        # fp32 training of a small model (gradient checks, ablations in full precision).
        _attn("f32_1500_gated_train", "train", "f32", 2, 4, 2, 1500, 64, 128),
        # The projection gates of a pre-training batch: 16 heads of 64, 16 sequences of 2048.
        _gates("gates_32768x1024_train", "bf16", 32768, 1024, True),
        # Prefill with rotary positions, token-major.
        _attn("rope_8192_gated", "rope", "bf16", 1, 32, 8, 8192, 128, 1024, layout="bnhd"),
        # Offloaded activations: Q, K, V come from and Y goes to pinned host memory.
        _attn("host_8192_gated", "host", "bf16", 1, 32, 8, 8192, 128, 1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# (heads, KV heads, head dimension): multi-head and grouped shapes of the configurations and tests
_HEADS = [(1, 1, 64), (4, 2, 64), (12, 12, 64), (16, 16, 64), (6, 2, 128), (8, 2, 128),
          (16, 16, 128), (32, 8, 128), (32, 4, 128)]


def draw(rng):
    kind = rng.choice(["forward", "gated", "gated", "rope", "train", "train", "train", "gates",
                       "host"])
    if kind == "gates":
        dm = rng.choice([512, 768, 1024, 2048, 4096])
        return _gates(None, "bf16", _log_int(rng, 1000, min(32768, 2.5e11 / dm ** 2)), dm,
                      rng.random() < 0.7)
    f32 = kind in ("forward", "gated", "train") and rng.random() < 0.2
    Hq, Hkv, d = rng.choice(_HEADS)
    if f32:
        # full precision: small models and checks
        n, B = _log_int(rng, 200, 2000), rng.choice([1, 2])
        Hq, Hkv = min(Hq, 8), min(Hkv, 2) if Hkv != Hq else min(Hkv, 8)
        w = _log_int(rng, 16, min(256, n))
    else:
        top = {"forward": 65536, "gated": 131072, "rope": 32768, "train": 16384, "host": 16384}[kind]
        n = _log_int(rng, 300, top)
        w = _log_int(rng, 32, min(2048, n))
        # tokens of a batch: what a prefill (few sequences) or a training batch (many) carries
        most = (65536 if kind == "train" else 32768) // n
        B = rng.randint(1, max(1, min(16, most)))
    causal = rng.random() < 0.85
    linear = rng.random() < 0.2
    layout = rng.choice(["bhnd", "bnhd"]) if kind != "host" else "bhnd"
    gated = kind in ("gated", "rope", "host") or (kind == "train" and rng.random() < 0.6)
    c = _attn(None, kind, "f32" if f32 else "bf16", B, Hq, Hkv, n, d, w, causal, linear, layout,
              gated)
    # never more than the largest listed case
    top = work(_attn("", "gated", "bf16", 1, 32, 4, 131072, 128, 2048))["flops"]
    while work(c)["flops"] > top / 2:
        c["n"] = max(300, c["n"] * 2 // 3)
        c["w"] = min(c["w"], c["n"])
    return c


def _flags(c):
    f = (sa.CAUSAL if c["causal"] else 0) | (sa.LINEAR_WINDOW if c["linear"] else 0)
    return f | (sa.SWA_ONE_SIDED if c["causal"] else 0)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def prepare(case, seed):
    c, g = case, _generator(seed)
    dt = DTYPES[c["dtype"]]
    normal = lambda *shape, scale=1.0: (torch.randn(*shape, generator=g, device="cuda") * scale).to(dt)
    s = {"case": c, "seed": seed}
    if c["kind"] == "gates":
        rows, dm = c["rows"], c["dm"]
        paths = 2 if c["dual"] else 1
        s["y"] = [normal(rows, dm) for _ in range(paths)]
        s["w"] = [normal(dm, dm, scale=dm ** -0.5) for _ in range(paths)]
        s["dout"] = normal(rows, dm)
        s["out"] = torch.empty(rows, dm, dtype=dt, device="cuda")
        return s
    B, Hq, Hkv, n, d = c["B"], c["Hq"], c["Hkv"], c["n"], c["d"]

    def heads(H):
        if c["layout"] == "bnhd":
            return normal(B, n, H, d).permute(0, 2, 1, 3)
        return normal(B, H, n, d)

    s["q"], s["k"], s["v"] = heads(Hq), heads(Hkv), heads(Hkv)
    s["flags"] = _flags(c)
    s["logits"] = torch.randn(2, Hq, generator=g, device="cuda")
    if c["kind"] == "host":
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)
        for name in ("q", "k", "v", "logits"):
            s[name] = pin(s[name])
        s["y"] = torch.empty(B, Hq, n, d, dtype=dt, pin_memory=True)
        s["host"] = HostForward(B, Hq, Hkv, n, d, c["w"], s["flags"], dtype=dt)
        return s
    if c["kind"] == "train":
        s["dy"] = heads(Hq)
    if c["kind"] == "rope":
        s["cos"], s["sin"] = sa.sa_rope_table(n, d, 1e6)
    if c["kind"] == "gated":
        # scratch that a serving program keeps from layer to layer
        p = sa.make_problem(s["q"], s["k"], c["w"], s["flags"])
        s["ws"] = torch.empty(sa.sa_workspace_bytes(p, sa.OP_GATED_FORWARD_SCRATCH),
                              dtype=torch.uint8, device="cuda")
    return s


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "gates":
        y, w = s["y"], s["w"]
        if c["dual"]:
            out = sa.sa_gate_projection_forward(y[0], w[0], y[1], w[1], out=s["out"])
            return (out,) + sa.sa_gate_projection_backward(s["dout"], y[0], w[0], y[1], w[1])
        out = sa.sa_gate_projection_forward(y[0], w[0], out=s["out"])
        return (out,) + sa.sa_gate_projection_backward(s["dout"], y[0], w[0])
    if kind == "host":
        return s["host"].forward(s["q"], s["k"], s["v"], s["logits"], s["y"], s["seed"], 0)
    q, k, v, w, flags = s["q"], s["k"], s["v"], c["w"], s["flags"]
    perm, inv = sa.sa_make_perm(s["seed"], 0, c["B"], c["n"])
    if kind == "forward":
        return perm, inv, sa.sa_forward(q, k, v, perm, inv, w, flags & ~sa.SWA_ONE_SIDED)
    if kind == "gated":
        return perm, inv, sa.sa_swa_gated_forward(q, k, v, perm, inv, s["logits"], w, flags,
                                                  ws=s["ws"])
    if kind == "rope":
        return perm, inv, sa.sa_swa_gated_forward_rope(q, k, v, perm, inv, s["cos"], s["sin"],
                                                       s["logits"], w, flags)
    if c["gated"]:
        saved = sa.sa_swa_gated_forward(q, k, v, perm, inv, s["logits"], w, flags, save_for_bwd=True)
        y, y_sa, y_swa, lse_sa, lse_swa = saved
        grads = sa.sa_backward(q, k, v, perm, inv, s["logits"], y_sa, y_swa, lse_sa, lse_swa,
                               s["dy"], w, flags)
        return (perm, inv) + tuple(saved) + tuple(grads)
    y, lse = sa.sa_forward(q, k, v, perm, inv, w, flags & ~sa.SWA_ONE_SIDED, want_lse=True)
    grads = sa.sa_backward(q, k, v, perm, inv, None, y, None, lse, None, s["dy"], w,
                           flags & ~sa.SWA_ONE_SIDED)
    return (perm, inv, y, lse) + tuple(grads[:3])


def _pairs(c, swa):
    """Visible (query, key) pairs of one head, per sequence (expected value for a random permutation
    with the linear window)."""
    n, w = c["n"], c["w"]
    if swa and c["causal"]:                       # one-sided: 0 <= i - j <= w - 1
        m = min(w, n)
        return n * m - m * (m - 1) / 2
    h = (w + 1) // 2 - 1
    if c["linear"]:
        m = min(h, n - 1)
        band = n + 2 * (n * m - m * (m + 1) / 2)
    else:
        band = n * min(n, 2 * h + 1)
    return n + (band - n) / 2 if c["causal"] else band


def work(case):
    """Each input read once, each output written once; two operations per multiply-add over the
    visible pairs: two products forward, five backward."""
    c = case
    elt = 2 if c["dtype"] == "bf16" else 4
    if c["kind"] == "gates":
        paths, rows, dm = (2 if c["dual"] else 1), c["rows"], c["dm"]
        forward = paths * (rows * dm + dm * dm) + rows * dm
        backward = paths * (2 * rows * dm + 2 * dm * dm) + rows * dm
        return {"bytes": (forward + backward) * elt, "flops": 4 * paths * 2.0 * rows * dm * dm}
    B, Hq, Hkv, n, d = c["B"], c["Hq"], c["Hkv"], c["n"], c["d"]
    qb, kb, rowf = B * Hq * n * d * elt, B * Hkv * n * d * elt, B * Hq * n * 4
    pairs = B * Hq * (_pairs(c, False) + (_pairs(c, True) if c["gated"] else 0))
    flops = 4.0 * pairs * d
    total = 2 * qb + 2 * kb + 2 * B * n * 4               # q, y, k, v, permutation and inverse
    if c["kind"] == "rope":
        total += n * d * 4
    if c["kind"] == "train":
        branches = 2 if c["gated"] else 1
        flops *= 3.5
        total += branches * rowf + (2 * qb if c["gated"] else 0)                 # saved state out
        total += qb * (1 + branches) + 2 * kb + branches * rowf + qb             # it, q, k, v, dy in
        total += qb + 2 * kb                                                     # dq, dk, dv out
    return {"bytes": float(total), "flops": flops}


def tolerance(case):
    return {"rel": 1e-2} if case["dtype"] == "bf16" else {"rel": 1e-5}

"""Workloads of the attention library: what its users run, at the sizes they run it.

A case is one training step (forward and backward) or one forward call of a transformer's attention,
through the entry points of ``paper_2608_01563_b200.binding``.  Sizes and value distributions are those
of ``paper_2608_01563_b200/inputs.py`` and of the tests.  Keys of a case:

family   "attn"   attention alone; ``pass`` says which calls:
                  "train"          forward + backward
                  "deterministic"  forward + the backward without floating-point atomics
                  "accel"          f16-product forward on f32 tensors + strict f32 backward
                  "forward"        forward only (prefill, chunked continuation, decode)
         "layer"  the whole attention layer: QKV projection with rotary embedding, attention, output
                  projection, and the backward of all three
mode     "strict" (f32 tensors) or "fast" (bf16 tensors)
B, H, Hkv, Sq, Sk, D, causal, and E (model width) for a layer
std      standard deviation of Q, K, V;  outliers: 1 % of the entries of Q and K scaled by 8
"""
from __future__ import annotations

import math

import torch

from paper_2608_01563_b200 import binding as mgn


def _attn(name, kind, mode, B, H, Hkv, Sq, Sk, D, causal, std=1.0, outliers=False):
    c = {"family": "attn", "pass": kind, "mode": mode, "B": B, "H": H, "Hkv": Hkv, "Sq": Sq, "Sk": Sk, "D": D,
         "causal": causal, "std": std, "outliers": outliers}
    if name:
        c["name"] = name
    return c


def _layer(name, B, H, Hkv, S, D, E):
    c = {"family": "layer", "pass": "train", "mode": "fast", "B": B, "H": H, "Hkv": Hkv, "Sq": S, "Sk": S, "D": D,
         "E": E, "causal": True, "std": 1.0, "outliers": False}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: two heads of 64 tokens; launches and latency
        _attn("tiny_strict_train", "train", "strict", 1, 2, 2, 64, 64, 32, False),
        # a GPT-2-small layer in f32 training: the default workload of bench.py
        _attn("gpt2_small_strict_train", "train", "strict", 8, 12, 12, 1024, 1024, 64, True, std=0.5),
        # a ViT-B layer in f32 training: 197 tokens is not a multiple of any tile
        _attn("vit_b_ragged_strict_train", "train", "strict", 32, 12, 12, 197, 197, 64, False),
        # a decoder block in f32 training, heavy-tailed scores
        _attn("decoder_s1024_strict_train", "train", "strict", 4, 32, 32, 1024, 1024, 128, True, outliers=True),
        # the accelerated policy on the GPT-2-small layer: f16 products forward, f32 backward
        _attn("gpt2_small_accel_train", "accel", "strict", 8, 12, 12, 1024, 1024, 64, True, std=0.5),
        # action tokens over a short context, many small heads
        _attn("cross_attn_action_fast_train", "train", "fast", 64, 8, 8, 50, 16, 64, False),
        # latent pixels over 77 text tokens: cross-attention of an image model
        _attn("cross_attn_text_fast_train", "train", "fast", 16, 8, 8, 1024, 77, 64, False),
        # a decoder block in bf16, reproducible from run to run
        _attn("decoder_s1024_fast_deterministic", "deterministic", "fast", 4, 32, 32, 1024, 1024, 128, True, outliers=True),
        # long-context bf16 training: the fast default of bench.py
        _attn("long_context_fast_train", "train", "fast", 2, 16, 16, 4096, 4096, 128, True),
        # the largest: a decoder block in bf16 training at 8192 tokens
        _attn("decoder_s8192_fast_train", "train", "fast", 4, 32, 32, 8192, 8192, 128, True, outliers=True),
        # inference: 512 new tokens at the end of a 4096-token context, grouped key/value heads
        _attn("gqa_suffix_fast_forward", "forward", "fast", 2, 16, 4, 512, 4096, 128, True),
        # a whole attention layer in bf16 training
        _layer("layer_s4096_fast_train", 2, 16, 16, 4096, 128, 2048),
    ]


def _log_int(rng, lo, hi):
    """Integer spread over the logarithm of [lo, hi], odd values as likely as even ones."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# the most a drawn case may cost, in floating-point operations: the strict cases run at an order of
# magnitude less per second, so they have a limit of their own
_LIMIT = {"strict": 1.5e11, "fast": 4.0e12}


def draw(rng):
    family = rng.choice(["strict_train", "strict_ragged", "strict_decoder", "strict_deterministic", "accel",
                         "cross", "fast_train", "fast_deterministic", "suffix", "suffix", "layer"])
    while True:
        if family in ("strict_train", "strict_deterministic"):
            s = _log_int(rng, 16, 4096)
            c = _attn(None, "train" if family == "strict_train" else "deterministic", "strict", rng.randint(1, 8),
                      rng.choice([2, 6, 12, 16]), 0, s, s, rng.choice([32, 64, 64, 128]), rng.random() < 0.6, std=0.5)
        elif family == "strict_ragged":
            s = _log_int(rng, 50, 600)
            c = _attn(None, "train", "strict", rng.randint(1, 32), 12, 0, s, s, 64, False)
        elif family == "strict_decoder":
            s = _log_int(rng, 128, 2048)
            c = _attn(None, rng.choice(["train", "forward"]), "strict", rng.randint(1, 4), rng.choice([8, 16, 32]), 0, s, s,
                      128, True, outliers=True)
        elif family == "accel":
            s = _log_int(rng, 64, 2048)
            c = _attn(None, "accel", "strict", rng.randint(1, 8), 12, 0, s, s, rng.choice([64, 128]), rng.random() < 0.6,
                      std=0.5)
        elif family == "cross":
            c = _attn(None, "train", "fast", rng.randint(1, 64), rng.choice([8, 16]), 0, _log_int(rng, 16, 2048),
                      _log_int(rng, 8, 320), rng.choice([64, 128]), False)
        elif family in ("fast_train", "fast_deterministic"):
            s = _log_int(rng, 64, 8192)
            c = _attn(None, "train" if family == "fast_train" else "deterministic", "fast", rng.randint(1, 4),
                      rng.choice([8, 16, 32]), 0, s, s, rng.choice([64, 128, 128]), rng.random() < 0.7,
                      outliers=rng.random() < 0.5)
        elif family == "suffix":
            sk = _log_int(rng, 256, 16384)
            c = _attn(None, "forward", rng.choice(["fast", "fast", "strict"]), rng.randint(1, 8), rng.choice([16, 32]), 0,
                      min(sk, _log_int(rng, 1, 1024)), sk, rng.choice([64, 128, 128]), True)
        else:
            H = rng.choice([8, 16])
            c = _layer(None, rng.randint(1, 4), H, rng.choice([H, H // 4]), _log_int(rng, 128, 4096),
                       rng.choice([64, 128]), 0)
            c["E"] = c["H"] * c["D"]
        if c["Hkv"] == 0:
            c["Hkv"] = c["H"] // 4 if family == "suffix" or (family == "fast_train" and rng.random() < 0.3) else c["H"]
        if c["family"] == "layer" and work(c)["flops"] > 1.3e12:
            continue
        if work(c)["flops"] <= _LIMIT[c["mode"]]:
            return c


# ---------------------------------------------------------------------------------------------------
def _scale(case):
    return 1.0 / math.sqrt(case["D"])


def _inputs(case, seed):
    """Inputs of a case, drawn on the GPU from the seed alone, in the element type of its mode."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float32 if case["mode"] == "strict" else torch.bfloat16

    def normal(*shape, std=1.0):
        t = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
        return t.mul_(std) if std != 1.0 else t

    B, H, Hkv, Sq, Sk, D = (case[n] for n in ("B", "H", "Hkv", "Sq", "Sk", "D"))
    if case["family"] == "layer":
        E, N = case["E"], (H + 2 * Hkv) * D
        x = normal(B, Sq, E).to(dt)
        w_qkv = normal(N, E, std=E ** -0.5).to(dt)
        w_o = normal(H * D, E, std=(H * D) ** -0.5).to(dt)
        d_y = normal(B, Sq, E).to(dt)
        angle = (torch.arange(Sq, device="cuda", dtype=torch.float64)[:, None]
                 * torch.pow(10000.0, -torch.arange(D // 2, device="cuda", dtype=torch.float64) / (D // 2)))
        return {"x": x, "w_qkv": w_qkv, "w_o": w_o, "d_y": d_y, "cos": angle.cos().float(), "sin": angle.sin().float()}
    q = normal(B, H, Sq, D, std=case["std"])
    k = normal(B, Hkv, Sk, D, std=case["std"])
    v = normal(B, Hkv, Sk, D, std=case["std"])
    if case["outliers"]:
        for t in (q, k):
            t[torch.rand(t.shape, generator=g, device="cuda") < 0.01] *= 8.0
    out = {"q": q.to(dt), "k": k.to(dt), "v": v.to(dt)}
    if case["pass"] != "forward":
        out["d_o"] = normal(B, H, Sq, D).to(dt)
    return out


def prepare(case, seed):
    st = {"case": case, "scale": _scale(case),
          "mode": mgn.MODE_STRICT_F32 if case["mode"] == "strict" else mgn.MODE_FAST_BF16}
    st.update(_inputs(case, seed))
    B, H, Hkv, Sq, Sk, D = (case[n] for n in ("B", "H", "Hkv", "Sq", "Sk", "D"))
    dt = torch.float32 if case["mode"] == "strict" else torch.bfloat16

    def empty(*shape, dtype=dt):
        return torch.empty(shape, device="cuda", dtype=dtype)

    st["o"], st["lse"] = empty(B, H, Sq, D), empty(B, H, Sq, dtype=torch.float32)
    if case["pass"] != "forward":
        st["dq"], st["dk"], st["dv"] = empty(B, H, Sq, D), empty(B, Hkv, Sk, D), empty(B, Hkv, Sk, D)
        st["ws"] = mgn.alloc_workspace(B, H, Sq, D, st["mode"])
    if case["pass"] == "accel":
        st["ws_fwd"] = empty(mgn.mgn_attn_fwd_accel_workspace_bytes(B, H, Hkv, Sq, Sk, D), dtype=torch.uint8)
    if case["family"] == "layer":
        E = case["E"]
        st["q"], st["k"], st["v"] = empty(B, H, Sq, D), empty(B, Hkv, Sk, D), empty(B, Hkv, Sk, D)
        st["y"], st["d_o"], st["delta"] = empty(B, Sq, E), empty(B, H, Sq, D), empty(B, H, Sq, dtype=torch.float32)
        st["d_x"], st["d_wqkv"], st["d_wo"] = empty(B, Sq, E), empty((H + 2 * Hkv) * D, E), empty(H * D, E)
    return st


def run(s):
    case = s["case"]
    causal, scale, mode = case["causal"], s["scale"], s["mode"]
    if case["family"] == "layer":
        mgn.mgn_qkv_rope_fwd(s["x"], s["w_qkv"], s["cos"], s["sin"], s["q"], s["k"], s["v"], mode)
        mgn.mgn_attn_fwd_ext(s["q"], s["k"], s["v"], s["o"], s["lse"], causal, scale, mode)
        mgn.mgn_out_proj_fwd(s["o"], s["w_o"], s["y"], mode)
        mgn.mgn_out_proj_bwd_weight(s["o"], s["d_y"], s["d_wo"], mode)
        mgn.mgn_out_proj_bwd_data(s["d_y"], s["w_o"], s["o"], s["d_o"], s["delta"], mode)
        mgn.mgn_attn_bwd_given_delta(s["q"], s["k"], s["v"], s["d_o"], s["lse"], s["delta"], s["dq"], s["dk"], s["dv"],
                                     s["ws"], causal, scale, mode)
        mgn.mgn_rope_bwd_inplace(s["dq"], s["dk"], s["cos"], s["sin"], mode)
        mgn.mgn_qkv_bwd_data(s["dq"], s["dk"], s["dv"], s["w_qkv"], s["d_x"], mode)
        mgn.mgn_qkv_bwd_weight(s["dq"], s["dk"], s["dv"], s["x"], s["d_wqkv"], mode)
        return {n: s[n] for n in ("y", "lse", "d_x", "d_wqkv", "d_wo")}
    square = case["H"] == case["Hkv"] and case["Sq"] == case["Sk"]
    if case["pass"] == "accel":
        mgn.mgn_attn_fwd_accel(s["q"], s["k"], s["v"], s["o"], s["lse"], s["ws_fwd"], causal, scale)
    elif square:
        mgn.mgn_attn_fwd(s["q"], s["k"], s["v"], s["o"], s["lse"], causal, scale, mode)
    else:
        mgn.mgn_attn_fwd_ext(s["q"], s["k"], s["v"], s["o"], s["lse"], causal, scale, mode)
    if case["pass"] == "forward":
        return {"o": s["o"], "lse": s["lse"]}
    bwd = (mgn.mgn_attn_bwd_deterministic if case["pass"] == "deterministic"
           else mgn.mgn_attn_bwd if square else mgn.mgn_attn_bwd_ext)
    bwd(s["q"], s["k"], s["v"], s["o"], s["d_o"], s["lse"], s["dq"], s["dk"], s["dv"], s["ws"], causal, scale, mode)
    return {n: s[n] for n in ("o", "lse", "dq", "dk", "dv")}


def work(case):
    B, H, Hkv, Sq, Sk, D = (case[n] for n in ("B", "H", "Hkv", "Sq", "Sk", "D"))
    e = 4 if case["mode"] == "strict" else 2
    # visible (query, key) pairs of a head: all, or keys j <= i + (Sk - Sq)
    pairs = Sq * (Sk - Sq) + Sq * (Sq + 1) / 2.0 if case["causal"] else float(Sq) * Sk
    nq, nk, rows = B * H * Sq * D, B * Hkv * Sk * D, B * H * Sq
    products = 4.0 if case["pass"] == "forward" else 14.0
    flops = products * B * H * pairs * D
    if case["family"] == "layer":
        E, N = case["E"], (H + 2 * Hkv) * D
        flops += 2.0 * B * Sq * E * 3 * (N + H * D)
        nbytes = e * (4 * B * Sq * E + 2 * N * E + 2 * H * D * E) + 4 * rows + 4 * Sq * D
    elif case["pass"] == "forward":
        nbytes = e * (2 * nq + 2 * nk) + 4 * rows
    else:                                    # reads q, k, v, dO; writes o, lse, dq, dk, dv
        nbytes = e * (4 * nq + 4 * nk) + 4 * rows
    return {"bytes": int(nbytes), "flops": float(flops)}


def tolerance(case):
    # f32 sums over up to 8192 terms with scores up to +-64; bf16 operands and results; for the
    # accelerated policy the f16 rounding of the forward's inputs
    if case["mode"] == "fast":
        return {"rel": 1.6e-2}
    if case["pass"] == "accel":
        return {"rel": 1.2e-3}
    return {"rel": 7e-6}


# ---------------------------------------------------------------------------------------------------
def _exact_attention(q, k, v, d_o, causal, scale):
    """(o, lse, dq, dk, dv) of one f64 head [S, D]; the last three are None without d_o."""
    s = (q @ k.T).mul_(scale)
    if causal:
        i = torch.arange(s.shape[0], device=s.device)[:, None] + (s.shape[1] - s.shape[0])
        s.masked_fill_(torch.arange(s.shape[1], device=s.device)[None, :] > i, -math.inf)
    lse = torch.logsumexp(s, dim=1)
    p = s.sub_(lse[:, None]).exp_()
    o = p @ v
    if d_o is None:
        return o, lse, None, None, None
    dv = p.T @ d_o
    ds = (d_o @ v.T).sub_((o * d_o).sum(1, keepdim=True)).mul_(p)
    return o, lse, (ds @ k).mul_(scale), (ds.T @ q).mul_(scale), dv


def _exact_heads(q, k, v, d_o, causal, scale):
    B, H, Sq, D = q.shape
    group = H // k.shape[1]
    f64 = {"device": q.device, "dtype": torch.float64}
    o, lse = torch.empty(q.shape, **f64), torch.empty(q.shape[:3], **f64)
    dq, dk, dv = torch.empty(q.shape, **f64), torch.zeros(k.shape, **f64), torch.zeros(k.shape, **f64)
    for b in range(B):
        for h in range(H):
            r = _exact_attention(q[b, h].double(), k[b, h // group].double(), v[b, h // group].double(),
                                 None if d_o is None else d_o[b, h].double(), causal, scale)
            o[b, h], lse[b, h] = r[0], r[1]
            if d_o is not None:
                dq[b, h] = r[2]
                dk[b, h // group] += r[3]
                dv[b, h // group] += r[4]
    return o, lse, dq, dk, dv


def exact(case, seed):
    if work(case)["flops"] > 2.0e13:
        return None
    t = _inputs(case, seed)
    causal, scale = case["causal"], _scale(case)
    if case["family"] == "attn":
        o, lse, dq, dk, dv = _exact_heads(t["q"], t["k"], t["v"], t.get("d_o"), causal, scale)
        if case["pass"] == "forward":
            return {"o": o, "lse": lse}
        return {"o": o, "lse": lse, "dq": dq, "dk": dk, "dv": dv}
    B, H, Hkv, S, D, E = (case[n] for n in ("B", "H", "Hkv", "Sq", "D", "E"))
    x, w_qkv, w_o, d_y = (t[n].double() for n in ("x", "w_qkv", "w_o", "d_y"))
    cos, sin = t["cos"].double(), t["sin"].double()

    def rotate(a, sign):                             # pairs (d, d + D/2) by the position's angles
        lo, hi = a[..., :D // 2], a[..., D // 2:]
        return torch.cat([lo * cos - sign * hi * sin, hi * cos + sign * lo * sin], dim=-1)

    def merge(a):                                    # [B,heads,S,D] -> [B*S, heads*D]
        return a.transpose(1, 2).reshape(B * S, -1)

    proj = (x.view(B * S, E) @ w_qkv.T).view(B, S, H + 2 * Hkv, D).transpose(1, 2)
    q, k, v = rotate(proj[:, :H], 1.0), rotate(proj[:, H:H + Hkv], 1.0), proj[:, H + Hkv:]
    d_o = (d_y.view(B * S, E) @ w_o.T).view(B, S, H, D).transpose(1, 2)
    o, lse, dq, dk, dv = _exact_heads(q, k, v, d_o, causal, scale)
    grad = merge(torch.cat([rotate(dq, -1.0), rotate(dk, -1.0), dv], dim=1))
    return {"y": (merge(o) @ w_o).view(B, S, E), "lse": lse, "d_x": (grad @ w_qkv).view(B, S, E),
            "d_wqkv": grad.T @ x.view(B * S, E), "d_wo": merge(o).T @ d_y.view(B * S, E)}

"""Timed cases of the boundary library: what a training program has it do, through the binding.

Every case is a dict with an "op":

  step      resbm_boundary_step: encode, decode, decode backward, encode backward of one pipeline
            boundary (the library's main path). T tokens of width d compressed to r, hidden width m
  host      resbm_boundary_step_host: the same step with its tensors in page-locked host memory
  send      resbm_ffn_down_encode_fwd: the FFN down-projection (width f to d) with the encoder fused
            in; F is stored too, since the encoder's backward reads it
  receive   the receiving block's start in training: resbm_decode_fwd_rmsnorm forward, then
            resbm_rmsnorm_bwd and resbm_decode_bwd
  muon      resbm_newton_schulz on the fp32 gradients of a boundary's four weights, five steps each
  rank      resbm_effective_rank of a bottleneck weight

Sizes: the shipped workloads (synth.CONFIGS, the pipeline's boundary) and the parity tests' ranges.
Inputs follow synth's recipe (activations N(0, 1) with a log-normal(0, 0.5) scale per token, weights
N(0, 1/fan_in)), drawn on the GPU from the seed.
"""
import math

import torch

from paper_2604_11947_gb300 import resbm

EPS = 1e-5
NS_STEPS = 5
DT = {"bf16": torch.bfloat16, "f32": torch.float32}
STEP_OPS = ("step", "host")
# One boundary's largest tensor (65536 x 4096) and largest product (32768 x 8192 x 512) of the shipped
# workloads bound what draw() gives; the portable kernels' cases are bounded like the tests'.
MOST_ELEMS = 65536 * 4096
MOST_PRODUCT = 32768 * 8192 * 512


def _step(name, T, d, r, m=None, **kw):
    case = {"name": name, "op": "step", "T": T, "d": d, "r": r, "m": r if m is None else m, "dtype": "bf16",
            "act": "silu", "merge": 1, "linear": False, "dX": True}
    case.update(kw)
    return case


def listed():
    return [
        # The smallest workload: batch 4 x seq 128, 128x compression, fp32 I/O. Latency and launches.
        _step("step_tiny_f32", 512, 256, 2, dtype="f32", dX=False),
        # A short ragged microbatch in bf16, with the options of reading (B): GELU, the pad added by the caller.
        _step("step_ragged", 1000, 512, 32, act="gelu_tanh", merge=0, dX=False),
        # One microbatch of the simulated pipeline: batch 8 x seq 2048, 128x.
        _step("step_single", 16384, 2048, 16),
        # The headline workload: batch 32 x seq 2048, 128x.
        _step("step_large", 65536, 4096, 32),
        # The compression sweep at d = 8192: 128x, 64x and 16x (compute-bound).
        _step("step_r64", 32768, 8192, 64),
        _step("step_r128", 32768, 8192, 128),
        _step("step_r512", 32768, 8192, 512),
        # A caller whose tensors live on the host: the pipeline's microbatch, both link directions.
        _step("host_single", 16384, 2048, 16, op="host", dX=False),
        # Sending stage of the pipeline: SwiGLU width 5632 down to d = 2048, encoded to r = 16.
        {"name": "send_ffn", "op": "send", "T": 16384, "f": 5632, "d": 2048, "r": 16, "m": 16, "act": "silu"},
        # Receiving stage of the pipeline in training: decoder + pre-attention norm, both backwards.
        {"name": "receive_norm", "op": "receive", "T": 16384, "d": 2048, "r": 16, "m": 16, "act": "silu", "merge": 1},
        # An optimizer step's orthogonalisation of the headline boundary's four weight gradients.
        {"name": "muon_r32", "op": "muon", "d": 4096, "r": 32, "m": 32},
        # The spectral analysis of the widest bottleneck projection.
        {"name": "rank_r512", "op": "rank", "rows": 8192, "cols": 512},
    ]


def _log_uniform(rng, lo, hi, multiple=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi, max(lo, int(round(v / multiple)) * multiple))


def _fit_tokens(rng, lo, hi, d, m):
    return _log_uniform(rng, lo, max(lo, min(hi, MOST_ELEMS // d, MOST_PRODUCT // (d * m))))


def _draw_step(rng, op):
    form = rng.choice(("fused", "fused", "fused", "widths", "portable"))
    if form == "fused":          # the widths of the workloads: m = r a power of two
        r = m = rng.choice((16, 32, 64, 128))
        d = _log_uniform(rng, max(256, r), 8192, 128)
        T, dtype = _fit_tokens(rng, 64, 65536, d, m), "bf16"
    elif form == "widths":       # any other bf16 widths, multiples of 8
        r, m = _log_uniform(rng, 8, 512, 8), _log_uniform(rng, 8, 512, 8)
        d = _log_uniform(rng, max(256, r), 8192, 8)
        T, dtype = _fit_tokens(rng, 64, 32768, d, max(r, m)), "bf16"
    else:                        # fp32, or odd widths
        r, m = _log_uniform(rng, 1, 32), _log_uniform(rng, 1, 32)
        d = _log_uniform(rng, 64, 1024)
        T, dtype = _log_uniform(rng, 64, 2048), rng.choice(("f32", "f32", "bf16"))
    if op == "host":
        T = min(T, max(64, (1 << 25) // d))
    linear = r == m and rng.random() < 0.15
    return {"op": op, "T": T, "d": d, "r": r, "m": m, "dtype": dtype,
            "act": rng.choice(("silu", "silu", "gelu_tanh", "identity")), "merge": rng.choice((1, 1, 0)),
            "linear": linear, "dX": op == "step" and rng.random() < 0.5}


def draw(rng):
    op = rng.choice(("step",) * 6 + ("host", "send", "receive", "receive", "muon", "rank"))
    if op in STEP_OPS:
        return _draw_step(rng, op)
    if op == "send":
        r, m = _log_uniform(rng, 4, 32), _log_uniform(rng, 8, 32, 8)
        d = _log_uniform(rng, 256, 4096, 8)
        f = _log_uniform(rng, 256, 11264, 8)
        return {"op": op, "T": _fit_tokens(rng, 64, 16384, max(d, f), 1), "f": f, "d": d, "r": r, "m": m,
                "act": rng.choice(("silu", "gelu_tanh"))}
    if op == "receive":
        r = m = rng.choice((16, 32, 64, 128))
        d = _log_uniform(rng, 256, 8192, 128)
        return {"op": op, "T": _fit_tokens(rng, 64, 32768, d, m), "d": d, "r": r, "m": m,
                "act": rng.choice(("silu", "gelu_tanh")), "merge": rng.choice((1, 0))}
    if op == "muon":
        r = _log_uniform(rng, 8, 512, 8)
        return {"op": op, "d": _log_uniform(rng, max(256, r), 8192, 8), "r": r, "m": rng.choice((r, _log_uniform(rng, 8, 512, 8)))}
    return {"op": op, "rows": _log_uniform(rng, 256, 8192, 8), "cols": _log_uniform(rng, 8, 512, 8)}


# ---- inputs ------------------------------------------------------------------------------------
def _randn(g, *shape, std=1.0):
    return torch.randn(*shape, generator=g, device="cuda").mul_(std)


def _inputs(case, seed):
    """The case's input tensors on the GPU, in their dtypes, from the seed alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    op = case["op"]
    if op == "rank":
        return {"W": _randn(g, case["rows"], case["cols"], std=case["rows"] ** -0.5).bfloat16()}
    d, r, m = case["d"], case["r"], case["m"]
    if op == "muon":   # fp32 weight gradients as the boundary step leaves them
        return {k: _randn(g, *s) for k, s in (("We1", (d, m)), ("We2", (m, r)), ("Wd1", (r, m)), ("Wd2", (m, d)))}
    T, io = case["T"], DT[case.get("dtype", "bf16")]
    scale = _randn(g, T, 1, std=0.5).exp_() if io == torch.bfloat16 else torch.ones(T, 1, device="cuda")
    h = {"We1": _randn(g, d, m, std=d ** -0.5), "We2": _randn(g, m, r, std=m ** -0.5),
         "Wd1": _randn(g, r, m, std=r ** -0.5), "Wd2": _randn(g, m, d, std=m ** -0.5)}
    h = {k: v.to(io) for k, v in h.items()}
    if op in STEP_OPS:
        h["X"] = _randn(g, T, d).mul_(scale).to(io)
        h["F"] = _randn(g, T, d).mul_(scale).to(io)
        h["dY"] = _randn(g, T, d).to(io)
        if case["dX"]:
            h["dX0"] = _randn(g, T, r).to(io)
        if case["linear"]:
            del h["We2"], h["Wd1"]
    elif op == "send":
        f = case["f"]
        h["X"] = _randn(g, T, d).mul_(scale).to(io)
        h["H"] = torch.nn.functional.silu(_randn(g, T, f)).mul_(_randn(g, T, f)).to(io)   # SwiGLU's hidden state
        h["W2"] = _randn(g, f, d, std=f ** -0.5).to(io)
        del h["Wd1"], h["Wd2"]
    else:   # receive
        h["B"] = _randn(g, T, r).mul_(scale).to(io)
        h["gamma"] = (1 + 0.1 * _randn(g, d)).to(io)
        h["dN"] = _randn(g, T, d).to(io)
        h["dY"] = _randn(g, T, d).to(io)
        del h["We1"], h["We2"]
    return h


def _desc(case):
    return resbm.make_desc(case["T"], case["d"], case["r"], case["m"], case.get("dtype", "bf16"), case["act"],
                           case.get("merge", 1), resbm.RESBM_FLAG_LINEAR if case.get("linear") else 0)


def prepare(case, seed):
    h = _inputs(case, seed)
    op = case["op"]
    s = {"case": case, "in": h}
    if op == "muon":
        s["out"] = {k: torch.empty_like(v, dtype=torch.bfloat16) for k, v in h.items()}
        s["ws"] = {k: resbm.matrix_workspace(resbm.RESBM_OP_NEWTON_SCHULZ, *v.shape) for k, v in h.items()}
        return s
    if op == "rank":
        s["out"] = torch.empty(4, dtype=torch.float64, device="cuda")
        s["ws"] = resbm.matrix_workspace(resbm.RESBM_OP_EFFECTIVE_RANK, *h["W"].shape)
        return s
    desc = s["desc"] = _desc(case)
    T, d, r, m = case["T"], case["d"], case["r"], case["m"]
    bf = {"dtype": torch.bfloat16, "device": "cuda"}
    f32 = {"dtype": torch.float32, "device": "cuda"}
    if op in STEP_OPS:
        out = resbm.step_outputs(desc, with_dX=case["dX"])
        if case["linear"]:
            del out["dWe2"], out["dWd1"]
        s["dX0"] = h.pop("dX0", None)
        if op == "step":
            s["ws"] = resbm.workspace(desc, resbm.RESBM_OP_BOUNDARY_STEP)
        else:
            s["ws"] = resbm.workspace(desc, resbm.RESBM_OP_BOUNDARY_STEP_HOST)
            s["in"] = {k: torch.empty(v.shape, dtype=v.dtype, pin_memory=True).copy_(v) for k, v in h.items()}
            out = {k: torch.zeros(v.shape, dtype=v.dtype, pin_memory=True) for k, v in out.items()}
        s["out"] = out
    elif op == "send":
        s["ws"] = resbm.ffn_down_encode_workspace(desc, case["f"])
        s["out"] = {"B": torch.empty(T, r, **bf), "P": torch.empty(T, m, **f32), "F": torch.empty(T, d, **bf)}
    else:
        s["ws"] = max((resbm.workspace(desc, o) for o in (resbm.RESBM_OP_DECODE_FWD_RMSNORM, resbm.RESBM_OP_RMSNORM_BWD,
                                                         resbm.RESBM_OP_DECODE_BWD)), key=torch.Tensor.numel)
        s["out"] = {"Y": torch.empty(T, d, **bf), "N": torch.empty(T, d, **bf), "dYs": torch.empty(T, d, **bf),
                    "dgamma": torch.empty(d, **f32), "dB": torch.empty(T, r, **bf), "dWd1": torch.empty(r, m, **f32),
                    "dWd2": torch.empty(m, d, **f32)}
    return s


def run(s):
    op, h, out, ws = s["case"]["op"], s["in"], s["out"], s["ws"]
    if op == "step":
        if s["dX0"] is not None:   # the residual gradient as the sending block's backward leaves it, r columns of it
            out["dX"][:, :s["dX0"].shape[1]].copy_(s["dX0"])
        resbm.resbm_boundary_step(s["desc"], ws, **h, **out)
    elif op == "host":
        resbm.resbm_boundary_step_host(s["desc"], ws, **h, **out)
    elif op == "send":
        resbm.resbm_ffn_down_encode_fwd(s["desc"], h["H"], h["W2"], h["X"], h["We1"], h["We2"], out["B"], out["P"],
                                        out["F"], ws)
    elif op == "receive":
        resbm.resbm_decode_fwd_rmsnorm(s["desc"], h["B"], h["Wd1"], h["Wd2"], h["gamma"], EPS, out["Y"], out["N"], ws)
        resbm.resbm_rmsnorm_bwd(s["desc"], out["Y"], h["gamma"], EPS, h["dN"], h["dY"], out["dYs"], out["dgamma"], ws)
        resbm.resbm_decode_bwd(s["desc"], out["dYs"], h["B"], h["Wd1"], h["Wd2"], out["dB"], out["dWd1"], out["dWd2"], ws)
    elif op == "muon":
        for k, G in h.items():
            resbm.resbm_newton_schulz(G, NS_STEPS, out[k], ws[k])
    else:
        resbm.resbm_effective_rank(h["W"], out, ws)
        # three results, each with an error of its own; the fourth word counts the method's iterations
        return {"sigma_max_sq": out[0], "fro_sq": out[1], "effective_rank": out[2]}
    return out


# ---- what a pass cannot do without ----------------------------------------------------------------
def work(case):
    op = case["op"]
    if op == "rank":
        n, k = max(case["rows"], case["cols"]), min(case["rows"], case["cols"])
        return {"bytes": 2 * n * k + 32, "flops": n * k * (k + 1)}   # the (symmetric) Gram matrix
    d, r, m = case["d"], case["r"], case["m"]
    if op == "muon":
        total = {"bytes": 0, "flops": 0}
        for a, b in ((d, m), (m, r), (r, m), (m, d)):
            n, k = max(a, b), min(a, b)
            total["bytes"] += 6 * a * b
            total["flops"] += NS_STEPS * (n * k * (k + 1) + 2 * k * k * k + 2 * n * k * k)
        return total
    T, e = case["T"], 4 if case.get("dtype") == "f32" else 2
    if op in STEP_OPS:
        w = d * m if case["linear"] else d * m + m * r
        lay = T * m * d if case["linear"] else T * m * (d + r)
        return {"bytes": e * T * (2 * d + r + 2 * d + 2 * r + (2 * r if case["dX"] else 0)) + 4 * T * m + 2 * w * (e + 4),
                "flops": 12 * lay}
    if op == "send":
        f = case["f"]
        return {"bytes": 2 * (T * f + f * d + T * r + d * m + m * r + T * r + T * d) + 4 * T * m,
                "flops": 2 * T * (f * d + d * m + m * r)}
    return {"bytes": 2 * (T * r + 2 * T * d + 3 * T * d + T * r) + 6 * (r * m + m * d + d),
            "flops": 2 * T * m * (d + r) * 3 + 8 * T * d}


def tolerance(case):
    op = case["op"]
    if op == "rank":       # fp32 Gram sums, the iteration stopped on a relative residual of 1e-5: up to 7e-7 seen
        return {"rel": 2e-5, "max": 2e-5}
    if op == "muon":       # bf16 iterates: 1.0-1.6e-2 seen against 64 bits, single elements up to 0.14 of the rms
        return {"rel": 3e-2, "max": 0.5}
    if case.get("dtype") == "f32":   # up to 8e-7 seen; sums over up to 2048 tokens in another order
        return {"rel": 1e-5, "max": 1e-4}
    # bf16 outputs, one rounding each (1.7e-3), and of operands rounded once before a product (up to 2.7e-3 seen)
    return {"rel": 1e-2, "max": 0.1}


# ---- the same in 64 bits ----------------------------------------------------------------------------
def _phi(case, x):
    if case["act"] == "identity" or case.get("linear"):
        return x
    if case["act"] == "silu":
        return x * torch.sigmoid(x)
    return 0.5 * x * (1 + torch.tanh(math.sqrt(2 / math.pi) * (x + 0.044715 * x ** 3)))


def _dphi(case, x):
    if case["act"] == "identity" or case.get("linear"):
        return torch.ones_like(x)
    if case["act"] == "silu":
        s = torch.sigmoid(x)
        return s * (1 + x * (1 - s))
    c = math.sqrt(2 / math.pi)
    t = torch.tanh(c * (x + 0.044715 * x ** 3))
    return 0.5 * (1 + t) + 0.5 * x * (1 - t * t) * c * (1 + 3 * 0.044715 * x * x)


def _decode_bwd(case, dY, B, Wd1, Wd2):
    """(dB, dWd1, dWd2); Wd1 None: one linear layer."""
    Q = B if Wd1 is None else B @ Wd1
    dWd2 = _phi(case, Q).T @ dY
    dQ = (dY @ Wd2.T) * _dphi(case, Q)
    dB = dQ if Wd1 is None else dQ @ Wd1.T
    if case["merge"]:
        dB = dB + dY[:, :case["r"]]
    return dB, None if Wd1 is None else B.T @ dQ, dWd2


def exact(case, seed):
    h = _inputs(case, seed)
    op = case["op"]
    if op == "rank":
        W = h["W"].double()
        lam = torch.linalg.eigvalsh(W.T @ W if W.shape[0] >= W.shape[1] else W @ W.T)[-1]
        return {"sigma_max_sq": lam, "fro_sq": W.square().sum(), "effective_rank": W.square().sum() / lam}
    if op == "muon":
        out = {}
        for k, G in h.items():
            X = G.double()
            tall = X.shape[0] > X.shape[1]
            X = X.T if tall else X
            X = X / (X.norm() + 1e-7)
            for _ in range(NS_STEPS):
                A = X @ X.T
                X = 3.4445 * X + (-4.7750 * A + 2.0315 * A @ A) @ X
            out[k] = X.T if tall else X
        return out
    io = DT[case.get("dtype", "bf16")]
    d, r = case["d"], case["r"]
    stored = lambda v: v.to(io).double()   # what crosses to the next op has the I/O type, as the op defines
    pad = lambda b: torch.nn.functional.pad(b, (0, d - r))
    dX0 = h.pop("dX0", None)
    X = h.pop("X")[:, :r].double() if "X" in h else None
    h = {k: v.double() for k, v in h.items()}
    if op == "send":
        F = h["H"] @ h["W2"]
        P = stored(F) @ h["We1"]
        return {"B": X + _phi(case, P) @ h["We2"], "P": P, "F": F}
    if op == "receive":
        B, gamma = h["B"], h["gamma"]
        Y = _phi(case, B @ h["Wd1"]) @ h["Wd2"]
        Y = Y + pad(B) if case["merge"] else Y
        Ys = stored(Y)
        s = (Ys.square().mean(1, keepdim=True) + EPS).rsqrt()
        dn = h["dN"] * gamma
        dYs = h["dY"] + s * dn - Ys * s ** 3 / d * (dn * Ys).sum(1, keepdim=True)
        dB, dWd1, dWd2 = _decode_bwd(case, stored(dYs), B, h["Wd1"], h["Wd2"])
        return {"Y": Y, "N": Y * s * gamma, "dYs": dYs, "dgamma": (h["dN"] * Ys * s).sum(0), "dB": dB, "dWd1": dWd1,
                "dWd2": dWd2}
    F, dY, We1, We2, Wd1, Wd2 = h["F"], h["dY"], h["We1"], h.get("We2"), h.get("Wd1"), h["Wd2"]
    P = F @ We1
    A = _phi(case, P)
    B = X + (A if We2 is None else A @ We2)
    Bs = stored(B)
    Y = _phi(case, Bs if Wd1 is None else Bs @ Wd1) @ Wd2
    if case["merge"]:
        Y = Y + pad(Bs)
    dB, dWd1, dWd2 = _decode_bwd(case, dY, Bs, Wd1, Wd2)
    dBs = stored(dB)
    dP = (dBs if We2 is None else dBs @ We2.T) * _dphi(case, P)
    out = {"B": B, "P": P, "Y": Y, "dB": dB, "dF": dP @ We1.T, "dWe1": F.T @ dP, "dWd2": dWd2}
    if not case["linear"]:
        out.update(dWe2=A.T @ dBs, dWd1=dWd1)
    if case["dX"]:
        out["dX"] = pad(dX0.double() + dBs)
    return out

"""The portable kernels of narrow bottlenecks (m, r <= 32) at the edges of their tiles: 16 tokens, 512
staged columns, 256 output columns, 64 gradient columns per cluster, the padded widths 4, 8, 16, 32, and
the first widths that take the wide kernels. Tolerances: the parity tests' (fp32 1e-5, bf16 2e-2)."""
import pytest
import torch

from gpu_helpers import gpu_step, host_inputs, oracle_step, to_dev
from paper_2604_11947_gb300 import resbm, synth
from test_parity_gpu import _compare_all

pytestmark = pytest.mark.gpu

# T, d, r, m
SHAPES = [(1, 1, 1, 1), (15, 64, 32, 4), (16, 512, 4, 32), (17, 513, 31, 5), (33, 255, 8, 8), (130, 1030, 4, 9),
          (2049, 65, 17, 16), (7, 257, 2, 17), (300, 70, 32, 32), (200, 96, 33, 32), (200, 96, 32, 33)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("T,d,r,m", SHAPES)
def test_narrow_step_matches_oracle(T, d, r, m, dtype):
    cfg = synth.BoundaryConfig("narrow_%d_%d_%d_%d" % (T, d, r, m), T=T, d=d, r=r, m=m, dtype=dtype,
                               act="gelu_tanh" if T % 2 else "silu", merge=T % 3 != 0)
    h = host_inputs(cfg)
    dev = {k: to_dev(v, cfg) for k, v in h.items()}
    flags = resbm.RESBM_FLAG_GENERIC
    got = gpu_step(cfg, dev, flags=flags)
    _compare_all(cfg, got, oracle_step(cfg, h), dev, flags)
    assert resbm.resbm_device_error() == 0


@pytest.mark.parametrize("T,d,r,m", [(65536, 64, 4, 4), (65536, 64, 16, 16), (65535, 40, 32, 31)])
def test_narrow_gradients_over_many_tokens(T, d, r, m):
    """fp32 weight gradients over a long run of tokens against 64 bits, on inputs with a mean (so that partial sums
    grow all along). A chain of n fp32 additions to a steadily growing sum has a relative error of about 2^-24 /
    sqrt(12) * sqrt(n / 3): 64-token blocks and their sums, n = 64 + 128, 1.4e-7; quarters of a rank's tokens, the
    d x m gradients, n = 2048, 4.5e-7 (less where the terms alternate). Bounds 2.5e-7 and 7e-7."""
    g = torch.Generator(device="cuda")
    g.manual_seed(T + r)
    rand = lambda *s: torch.randn(*s, generator=g, device="cuda")
    dev = {"X": rand(T, d), "F": rand(T, d) + 0.3, "dY": rand(T, d) + 0.3, "We1": rand(d, m) * d ** -0.5,
           "We2": rand(m, r) * m ** -0.5, "Wd1": rand(r, m) * r ** -0.5, "Wd2": rand(m, d) * m ** -0.5}
    desc = resbm.make_desc(T, d, r, m, "f32", "silu", 1, 0)
    o = resbm.step_outputs(desc)
    resbm.resbm_boundary_step(desc, resbm.workspace(desc, resbm.RESBM_OP_BOUNDARY_STEP), **dev, **o)
    h = {k: v.double() for k, v in dev.items()}
    sig = torch.sigmoid
    dphi = lambda x: sig(x) * (1 + x * (1 - sig(x)))
    P, B, dB = h["F"] @ h["We1"], o["B"].double(), o["dB"].double()
    Q = B @ h["Wd1"]
    dQ, dP = (h["dY"] @ h["Wd2"].T) * dphi(Q), (dB @ h["We2"].T) * dphi(P)
    want = {"dWe1": h["F"].T @ dP, "dWe2": (P * sig(P)).T @ dB, "dWd1": B.T @ dQ, "dWd2": (Q * sig(Q)).T @ h["dY"]}
    for k, w in want.items():
        err = float((o[k].double() - w).norm() / w.norm())
        assert err <= (2.5e-7 if k in ("dWe2", "dWd1") else 7e-7), (k, err)
    assert resbm.resbm_device_error() == 0

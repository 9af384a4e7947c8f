"""The choice between the fused kernels and the chain of products by size (both take these shapes): each
side of the lines against the oracle, and P recomputed in the encoder backward equal to the saved P's result
where the two ops take different paths. Tolerances: the parity tests'."""
import pytest
import torch

from gpu_helpers import gpu_step, host_inputs, oracle_step, to_dev
from paper_2604_11947_gb300 import resbm, synth
from test_parity_gpu import _compare_all

pytestmark = pytest.mark.gpu

# T, d, r = m
SHAPES = [(2048, 2048, 16), (2049, 2048, 16), (700, 1408, 16), (2048, 1024, 32), (2049, 1024, 32), (1000, 768, 32),
          (520, 2048, 64), (520, 1920, 64), (300, 256, 64), (260, 512, 128), (1024, 4096, 32), (1025, 4096, 32),
          (73729, 1024, 64), (77824, 1024, 64), (39000, 1024, 64), (19457, 2048, 64), (1000, 8192, 16),
          (6000, 4096, 16), (1, 512, 32), (8192, 2432, 32), (19500, 2432, 32), (58400, 2048, 64)]


@pytest.mark.parametrize("T,d,r", SHAPES)
def test_routes_match_oracle(T, d, r):
    cfg = synth.BoundaryConfig("route_%d_%d_%d" % (T, d, r), T=T, d=d, r=r, m=r)
    h = host_inputs(cfg)
    dev = {k: to_dev(v, cfg) for k, v in h.items()}
    got = gpu_step(cfg, dev)
    _compare_all(cfg, got, oracle_step(cfg, h), dev)
    # without the saved P
    desc = resbm.desc_from_config(cfg)
    dF, dWe1, dWe2 = torch.empty_like(got["dF"]), torch.empty_like(got["dWe1"]), torch.empty_like(got["dWe2"])
    resbm.resbm_encode_bwd(desc, got["dB"], dev["F"], None, dev["We1"], dev["We2"], dF, None, dWe1, dWe2,
                           resbm.workspace(desc, resbm.RESBM_OP_ENCODE_BWD))
    assert torch.equal(dF, got["dF"]) and torch.equal(dWe1, got["dWe1"]) and torch.equal(dWe2, got["dWe2"])
    assert resbm.resbm_device_error() == 0


@pytest.mark.parametrize("T,d,r", [(520, 2048, 64), (300, 256, 64), (260, 512, 128), (700, 1408, 16)])
def test_gradients_not_16_byte_aligned(T, d, r):
    """Weight gradients at a 4-byte aligned address: the same bits as aligned ones."""
    cfg = synth.BoundaryConfig("route_al_%d" % T, T=T, d=d, r=r, m=r)
    dev = {k: to_dev(v, cfg) for k, v in host_inputs(cfg).items()}
    want = gpu_step(cfg, dev)
    desc = resbm.desc_from_config(cfg)
    off = lambda t: torch.empty(t.numel() + 4, device="cuda")[1:1 + t.numel()].view(t.shape)
    dF, dWe1, dWe2 = torch.empty_like(want["dF"]), off(want["dWe1"]), off(want["dWe2"])
    resbm.resbm_encode_bwd(desc, want["dB"], dev["F"], want["P"], dev["We1"], dev["We2"], dF, None, dWe1, dWe2,
                           resbm.workspace(desc, resbm.RESBM_OP_ENCODE_BWD))
    assert torch.equal(dF, want["dF"]) and torch.equal(dWe1, want["dWe1"]) and torch.equal(dWe2, want["dWe2"])
    assert resbm.resbm_device_error() == 0


@pytest.mark.parametrize("cluster", ["1", "2"])
@pytest.mark.parametrize("T,d", [(1000, 512), (300, 192), (20000, 64)])
def test_fused_m64_matches_oracle(T, d, cluster, monkeypatch):
    """The fused m = 64 kernels at sizes that the chain takes by itself (a forced cluster size keeps them)."""
    monkeypatch.setenv("RESBM_CLUSTER", cluster)
    cfg = synth.BoundaryConfig("route_fused_%d_%d" % (T, d), T=T, d=d, r=64, m=64)
    h = host_inputs(cfg)
    dev = {k: to_dev(v, cfg) for k, v in h.items()}
    _compare_all(cfg, gpu_step(cfg, dev), oracle_step(cfg, h), dev)
    assert resbm.resbm_device_error() == 0


@pytest.mark.parametrize("T,d,r,encoder", [(33000, 512, 64, True), (16384, 4096, 64, True), (45000, 2048, 64, True),
                                           (1000, 4096, 64, True), (4096, 8192, 32, False)])   # (False: fused anyway)
def test_chain_sums_are_as_exact_as_the_fused_kernels(T, d, r, encoder, monkeypatch):
    """Where the chain replaces a fused kernel, the error of its long sums (P over d, the weight gradients of hi + lo
    operands over the tokens) against 64 bits is no larger than the fused kernel's (which a forced cluster size
    keeps): at most 1.05 of it, for the error's own spread from one order of summation to another (a few per cent of
    a 2-norm over at least 10^3 elements)."""
    cfg = synth.BoundaryConfig("route_err_%d_%d" % (T, d), T=T, d=d, r=r, m=r)
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    rand = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
    X, F, dY, B = rand(T, d), rand(T, d), rand(T, d), rand(T, r)
    We1, We2, Wd1, Wd2 = rand(d, r) * d ** -0.5, rand(r, r) * r ** -0.5, rand(r, r) * r ** -0.5, rand(r, d) * r ** -0.5
    desc = resbm.desc_from_config(cfg)
    ws = resbm.workspace(desc, resbm.RESBM_OP_BOUNDARY_STEP)
    D = torch.Tensor.double
    Q = D(B) @ D(Wd1)
    s = torch.sigmoid(Q)
    dQ = (D(dY) @ D(Wd2).T) * (s * (1 + Q * (1 - s)))
    want = {"dWd2": (Q * s).T @ D(dY), "dWd1": D(B).T @ dQ}
    if encoder:
        want["P"] = D(F) @ D(We1)

    def errors():
        o = resbm.step_outputs(desc)
        resbm.resbm_encode_fwd(desc, X, F, We1, We2, o["B"], o["P"], ws)
        resbm.resbm_decode_bwd(desc, dY, B, Wd1, Wd2, o["dB"], o["dWd1"], o["dWd2"], ws)
        return {k: float((D(o[k]) - w).norm() / w.norm()) for k, w in want.items()}

    chain = errors()
    monkeypatch.setenv("RESBM_CLUSTER", "4")
    fused = errors()
    for k in want:
        assert chain[k] <= 1.05 * fused[k], (k, chain, fused)
    assert resbm.resbm_device_error() == 0

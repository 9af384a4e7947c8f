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
          (6000, 4096, 16), (1, 512, 32), (8192, 2432, 32), (19500, 2432, 32)]


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

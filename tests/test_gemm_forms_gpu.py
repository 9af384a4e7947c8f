"""The GEMM chain's units on CTA pairs (two-CTA MMAs) against its single-CTA units (RESBM_GEMM_MC=0): the
per-token outputs bit for bit (every element summed over K in the same order), the weight gradients, whose
split count may differ, to fp32 accumulation in another order."""
import pytest
import torch

from gpu_helpers import gpu_step, host_inputs, to_dev
from paper_2604_11947_gb300 import resbm, synth

pytestmark = pytest.mark.gpu

# one row past a block, an odd number of row blocks (a pair's second CTA idle), ragged columns and K
SHAPES = [(129, 264, 136, 144), (257, 520, 264, 136), (385, 512, 256, 512), (700, 328, 320, 264)]


@pytest.mark.parametrize("T,d,r,m", SHAPES)
def test_pairs_match_single_ctas(T, d, r, m, monkeypatch):
    cfg = synth.BoundaryConfig("pairs_%d" % T, T=T, d=d, r=r, m=m)
    dev = {k: to_dev(v, cfg) for k, v in host_inputs(cfg).items()}
    flags = resbm.RESBM_FLAG_GEMM
    pairs = gpu_step(cfg, dev, flags=flags)
    monkeypatch.setenv("RESBM_GEMM_MC", "0")
    single = gpu_step(cfg, dev, flags=flags)
    for k in ("B", "P", "Y", "dB", "dF", "dX"):
        assert torch.equal(pairs[k], single[k]), k
    for k in ("dWe1", "dWe2", "dWd1", "dWd2"):
        err = (pairs[k] - single[k]).abs().max() / single[k].square().mean().sqrt()
        # sums of up to 700 terms, each partial rounded to 2^-24: sqrt(700) 2^-24 = 1.6e-6 of the RMS
        # for one element, six times that for the largest of 2.7e5: 1e-5, bound ten times it
        assert err <= 1e-4, (k, float(err))
    assert resbm.resbm_device_error() == 0


@pytest.mark.parametrize("T,d,r", [(19457, 1024, 128), (20011, 1032, 64), (38913, 1024, 40), (45000, 1024, 72)])
def test_row_balanced_units_match_whole_blocks(T, d, r, monkeypatch):
    """More row blocks than SMs and one column block: rows spread evenly over the CTAs (the last unit of each
    shorter), against 128-row blocks (RESBM_GEMM_TS=0, which also stores without TMA): the same bits."""
    cfg = synth.BoundaryConfig("rows_%d" % T, T=T, d=d, r=min(r, d), m=r)
    dev = {k: to_dev(v, cfg) for k, v in host_inputs(cfg).items()}
    flags = resbm.RESBM_FLAG_GEMM
    got = gpu_step(cfg, dev, flags=flags)
    monkeypatch.setenv("RESBM_GEMM_TS", "0")
    want = gpu_step(cfg, dev, flags=flags)
    for k in ("B", "P", "Y", "dB", "dF", "dX", "dWe1", "dWe2", "dWd1", "dWd2"):
        assert torch.equal(got[k], want[k]), k
    assert resbm.resbm_device_error() == 0


@pytest.mark.parametrize("T,d,m", [(300, 8192, 512), (260, 8168, 264), (192, 7424, 384)])
def test_narrower_gradient_tiles_match_single_ctas(T, d, m, monkeypatch):
    """Weight gradients whose tiles are narrowed to even out the last round of pairs (d x m and m x d, the last
    tile ragged), against single CTAs (RESBM_GEMM_MC=0): one split in both, so the same bits."""
    cfg = synth.BoundaryConfig("vn_%d" % d, T=T, d=d, r=m, m=m)
    dev = {k: to_dev(v, cfg) for k, v in host_inputs(cfg).items()}
    flags = resbm.RESBM_FLAG_GEMM
    got = gpu_step(cfg, dev, flags=flags)
    monkeypatch.setenv("RESBM_GEMM_MC", "0")
    want = gpu_step(cfg, dev, flags=flags)
    for k in ("dWe1", "dWd2", "dF", "Y"):
        assert torch.equal(got[k], want[k]), k
    assert resbm.resbm_device_error() == 0

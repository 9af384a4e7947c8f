"""The portable kernels of narrow bottlenecks (m, r <= 32) at the edges of their tiles: 16 tokens, 512
staged columns, 256 output columns, 64 gradient columns per cluster, the padded widths 4, 8, 16, 32, and
the first widths that take the wide kernels. Tolerances: the parity tests' (fp32 1e-5, bf16 2e-2)."""
import pytest

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

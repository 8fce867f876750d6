"""The FP64 rate probe reaches the pipe's own rate (GPU): a warp's fused multiply-add with its operands in
registers takes 64 cycles of the pipe, an add or a multiply 76."""
import pytest

from paper_2609_10816_gb300 import mhd

pytestmark = pytest.mark.gpu


def test_dfma_rate_is_the_pipes(gpu_lib):
    r = {k: mhd.fp64_rate(k, 1 << 13) for k in ("dfma", "dadd", "dmul", "dfma_16_lanes")}
    assert r["dfma"] > 1.1 * r["dadd"] and r["dfma"] > 1.1 * r["dmul"]
    assert 0.45 < r["dfma_16_lanes"] / r["dfma"] < 0.55

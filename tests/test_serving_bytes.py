"""The serving budget counts at least what a run adds to a batch's tile list:
an 8-byte record per 32 x 8 tile in FP32, per block of 64 nodes in FP64."""
import pytest

from paper_1608_01906_gb300 import serving


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("side", [32, 33, 64, 95, 333, 512, 1024])
def test_run_bytes_cover_the_tile_list(side, precision):
    records = -(-side // 32) * -(-side // 8) if precision == "fp32" else -(-side * side // 64)
    listed = serving.run_bytes(side, precision) - serving.state_bytes(side, precision) - serving.BATCH_RUN_BYTES
    assert listed >= 8 * records

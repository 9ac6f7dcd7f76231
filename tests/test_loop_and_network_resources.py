"""Register and local-memory budgets of the on-chip 2D loops and of the network's convolutions,
from ptxas's resource report (no GPU needed).

A loop's tile leaves the SM no L1, so a spill there is a round trip to L2 on every row: every
variant keeps its state in registers, at most 128 a thread (512 threads).  The convolutions run
three (16 input channels: four) blocks of 192 threads per SM; the one that sums the decoder's inputs
holds a coarse row in registers beside an accumulator row and spills up to 100 bytes, once a row of
128 pixels."""
import pytest

from test_kernel_resources import _ptxas_report, pytestmark  # noqa: F401


@pytest.mark.parametrize("src,kernels", [("fd2loop32.cu", 19), ("fd2loop64.cu", 19)])
def test_on_chip_loops_keep_their_state_in_registers(src, kernels, tmp_path):
    rows = {k: v for k, v in _ptxas_report(src, tmp_path).items() if "fd2_loop_kernel" in k}
    assert len(rows) == kernels, sorted(rows)
    for k, v in rows.items():
        assert v["stack"] == 0 and v["spill"] == 0 and v["regs"] <= 128, (k, v)


def test_convolutions_stay_within_their_register_budget(tmp_path):
    rows = {k: v for k, v in _ptxas_report("pc.cu", tmp_path).items() if "conv3x3_tc_kernel" in k}
    assert rows
    for k, v in rows.items():
        blocks = 4 if "ILi16E" in k else 3
        assert v["regs"] * 192 * blocks <= 65536, (k, v)
        assert v["spill"] <= 100, (k, v)

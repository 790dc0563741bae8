"""The check of the step kernel's register split before any launch: row warps
(8 of 12) take 96 or 88 registers, the other four keep 48 or 64, 80 a thread
on average, so a kernel compiled for fewer is refused on the host."""
import pytest

from paper_2207_06908_gb300 import _build, _lib


@pytest.mark.parametrize("regs,rc", [(80, 0), (88, 0), (255, 0), (79, -4), (72, -4), (1, -4), (0, -1), (256, -1)])
def test_split_needs_eighty(regs, rc):
    _build.build()
    assert _lib.load().fdtd_selftest_registers(regs) == rc

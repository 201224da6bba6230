"""The phase-clock diagnostic without a GPU: its patches apply to the kernel's
current source, its table is made of the recorded CTAs alone, and a shape whose
launch is not persistent (no CTA records anything) is an error that says so."""

import os

import numpy as np
import pytest

from paper_1104_3408_gb300 import _build, phase_clocks


def test_patches_apply_to_the_kernel():
    with open(os.path.join(_build.CSRC, "ops.cu")) as fh:
        src = fh.read()
    s = phase_clocks._patched_ops(src)
    assert "cffyn_instr_read" in s and s.count("g_instr[blockIdx.x]") == 3


def test_table_of_the_recorded_ctas():
    buf = np.zeros((1024, 16), dtype=np.uint64)
    buf[:3, :11] = 2000  # cycles
    buf[:3, 11] = 500
    buf[:3, 12] = 2      # items
    lines = phase_clocks.report(buf, (33, 48, 96), 1000.0).splitlines()
    assert "33x48x96" in lines[0] and "3 CTAs, 2.00 items" in lines[0]
    assert len(lines) == 1 + len(phase_clocks.NAMES)
    assert lines[1].split()[-3:] == ["1.00"] * 3 and lines[-1].split()[-3:] == ["0.50"] * 3


def test_no_records_is_an_error_that_names_the_shape():
    with pytest.raises(RuntimeError, match="9x12x24 shell has too few items"):
        phase_clocks.report(np.zeros((1024, 16), dtype=np.uint64), (9, 12, 24), 2070.0)

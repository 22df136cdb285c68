"""Registers of the kernels whose speed hangs on how many CTAs an SM holds, as
ptxas reports them.
"""
import re
import subprocess

import pytest

from paper_1208_6350_gb300 import _build


def usage(source, tmp_path):
    """{mangled kernel name: (registers, spilled bytes)} of one source file."""
    try:
        nvcc = _build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    r = subprocess.run([nvcc] + _build._flags() + ["-Xptxas", "-v", "-cubin", f"{_build.CSRC}/{source}", "-o",
                                                   str(tmp_path / "k.cubin")], capture_output=True, text=True, check=True)
    out = {}
    for part in r.stderr.split("Compiling entry function")[1:]:
        spill = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", part)
        out[part.split("'")[1]] = (int(re.search(r"Used (\d+) registers", part).group(1)),
                                   int(spill.group(1)) + int(spill.group(2)))
    return out


def test_wide_band_traceback_leaves_room_for_two_ctas(tmp_path):
    # 256 threads a CTA and 65,536 registers an SM: the 16-row form of batches of
    # more than 5,000 pairs, and the 8-row form
    kernels = {k: v for k, v in usage("trace_ring.cu", tmp_path).items() if "k_trace_ring" in k}
    two = {k: v for k, v in kernels.items() if "RingCfgILi8E" in k or "RingCfgILi16EEELi2E" in k}
    assert len(kernels) == 6 and len(two) == 4, kernels  # 4-letter or general alphabets
    for name, (registers, spilled) in two.items():
        assert registers <= 128 and spilled == 0, (name, registers, spilled)

"""What ptxas reports of kernels whose speed hangs on it: registers decide how many CTAs share an SM, and a spill in a loop
is paid on every trip."""
import os
import re
import subprocess

import pytest

from paper_2607_22595_b200 import _build

LIMITS = [
    # four CTAs of 256 threads per SM leave 64 registers.  What lives across a row's steps does not fit, with or without the
    # gather (88 bytes of spill stores before it read its lists in whole batches, 292 after): outside the loops, some 100 bytes.
    ("sae_tail.cu", "tail_kernel", 64, 112),
    # beside it two CTAs of the streaming kernel (72 registers a thread) are to fit into the SM's 64 Ki registers: at most 112,
    # and at the launch bound of three CTAs 80
    ("probe_tc.cu", "probe_tc_kernel", 80, 0),
]


@pytest.mark.parametrize("source,kernel,registers,spill_bytes", LIMITS)
def test_registers_and_spills(tmp_path, source, kernel, registers, spill_bytes):
    cmd = [_build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo", "-Xptxas", "-v", "-Xcompiler", "-fPIC",
           "-I", os.path.join(_build.ROOT, "include"), "-I", _build.CSRC, "-c", os.path.join(_build.CSRC, source), "-o", str(tmp_path / "kernel.o")]
    report = subprocess.run(cmd, capture_output=True, text=True, check=True).stderr
    entries = [e for e in report.split("Compiling entry function")[1:] if kernel in e.splitlines()[0]]
    assert entries, report
    for entry in entries:
        assert int(re.search(r"Used (\d+) registers", entry).group(1)) <= registers
        assert int(re.search(r"(\d+) bytes spill stores", entry).group(1)) <= spill_bytes

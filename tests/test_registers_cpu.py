"""Register budgets of the FP32 force pass: its launch bounds are set so that
the pair loop keeps its values in registers (a spilled one cost 5 % of a step),
in every variant, as the compiler reports them."""
import os
import re
import subprocess

from paper_2411_13992_gb300 import _build


def test_force_pass_spills_no_registers(tmp_path):
    cmd = [_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-Xptxas", "-v", "-c",
           os.path.join(_build.CSRC, "k_pair32.cu"), "-o", str(tmp_path / "k_pair32.o")]
    r = subprocess.run(cmd, capture_output=True, text=True, check=True)
    kernel, spills = None, {}
    for line in r.stderr.splitlines():
        m = re.search(r"Compiling entry function '(\w+)'", line)
        if m:
            kernel = m.group(1)
        m = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", line)
        if m:
            spills[kernel] = (int(m.group(1)), int(m.group(2)))
    forces = {k: v for k, v in spills.items() if "k_forces32" in k}
    assert len(forces) >= 12            # 2 and 3 dimensions, both kinds of sums, uniform (two depths) and varying h
    assert all(v == (0, 0) for v in forces.values()), forces

"""CPU: the register budgets of the force and near-field kernels, as the compiler reports them. They
are bound by latency and issue, so what a change of the shared stress code
spills shows in their times; the limits are what they were tuned with."""
import os
import re
import subprocess

import pytest

from paper_2003_03130_gb300 import build

# source, kernel, registers, bytes of spill stores
LIMITS = [("tet_force.cu", "k_tet_force", 40, 28), ("chain.cu", "k_cell_chain<2>", 64, 32), ("chain.cu", "k_cell_chain<4>", 64, 44),
          ("relax.cu", "k_relax_cells", 64, 0), ("relax.cu", "k_relax_reverse", 128, 0)]
LIMITS += [("lbm.cu", f"k_lbm_near<{t}, {keep}, true>", 64, 0) for t in ("float", "__half", "__nv_bfloat16") for keep in ("false", "true")]


def used(source):
    release = subprocess.run([build.nvcc(), "--version"], capture_output=True, text=True).stdout
    if "release 13.0" not in release:
        pytest.skip("the limits are those of nvcc 13.0")
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-Xptxas", "-v", "-c", os.path.join(build.CSRC, source), "-o",
                        os.devnull], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = {}
    for part in r.stderr.split("Compiling entry function '")[1:]:
        name = subprocess.run(["c++filt", part.split("'")[0]], capture_output=True, text=True).stdout
        name = name.split("(")[0].split("cf::")[-1]
        out[name] = int(re.search(r"Used (\d+) registers", part)[1]), int(re.search(r"(\d+) bytes spill stores", part)[1])
    return out


@pytest.mark.parametrize("source", sorted({k[0] for k in LIMITS}))
def test_registers_and_spills(source):
    got = used(source)
    for src, kernel, registers, spill in LIMITS:
        if src == source:
            assert got[kernel][0] <= registers and got[kernel][1] <= spill, (kernel, got[kernel])

"""Register budgets of the docking kernel's entry points beside those of test_kernel_resources.py, as ptxas reports them
(nvcc cross-compiles for sm_103a without a GPU, so this runs on the CPU): 80 registers with 2 warps per item on a
trilinear grid, 96 with one (on the integer grid with a pose tile of 2), the 64-register launch bound elsewhere."""
import os
import re
import subprocess
from concurrent.futures import ThreadPoolExecutor

import pytest

from paper_2209_05069_gb300 import build

ENTRY = re.compile(r"Compiling entry function '_ZN7dockgpu\d+(dock_kernel(?:_wide|_mid)?)ILi(\d+)E")
UNITS = {(0, 2, 1): ("dock_kernel_mid", 80), (1, 2, 2): ("dock_kernel_mid", 80), (1, 1, 2): ("dock_kernel_wide", 96),
         (2, 1, 2): ("dock_kernel_wide", 96), (2, 1, 1): ("dock_kernel", 64), (2, 2, 1): ("dock_kernel", 64),
         (0, 4, 1): ("dock_kernel", 64), (1, 4, 1): ("dock_kernel", 64)}   # (grid type, warps per item, pose tile)


def _compile(unit, out):
    gt, g, t = unit
    cmd = [build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", build.INCLUDE, "-I", build.CSRC,
                                         f"-DDOCK_INST_GT={gt}", f"-DDOCK_INST_G={g}", f"-DDOCK_INST_T={t}", "-Xptxas", "-v",
                                         "-c", os.path.join(build.CSRC, "dock_kernels_inst.cu"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    found, cur = {}, None
    for line in r.stderr.splitlines():
        m = ENTRY.search(line)
        if m:
            cur = m.group(1), int(m.group(2))
        m = re.search(r"Used (\d+) registers", line)
        if m and cur:
            found[cur] = int(m.group(1))
            cur = None
    return found


def test_entry_points_and_registers(tmp_path):
    try:
        build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    with ThreadPoolExecutor(max_workers=min(len(UNITS), os.cpu_count() or 4)) as ex:
        got = list(ex.map(lambda u: _compile(u, str(tmp_path / ("k%d%d%d.o" % u))), UNITS))
    for unit, found in zip(UNITS, got):
        entry, most = UNITS[unit]
        assert sorted(n for _, n in found) == [32, 64, 96, 128, 160], unit
        for (name, n), regs in found.items():
            assert name == entry and regs <= most, (unit, name, n, regs)

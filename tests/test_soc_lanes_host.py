"""Host-only check of the number of lanes that share one Lorentz cone (soc_lanes): the
widths that the cone tests on the GPU are named by, and the rule's limits."""
import os
import shutil
import subprocess

import pytest

from paper_2103_00736_gb300 import build

# cone sizes -> lanes
CASES = [([2], 4), ([2, 3, 4, 5, 31, 32, 33, 48], 4), ([48] * 5, 4), ([49] * 12, 8), ([96] * 3, 8), ([100] * 9, 16),
         ([200] * 7, 32), ([3] * 40 + [256], 4), ([3] * 40 + [300], 8), ([3] * 40 + [600], 16), ([3] * 40 + [2100], 32),
         ([2] * 1500, 4), ([100_000], 32)]


def test_widths(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "lanes.cu"
    src.write_text('#include "acs_host.cuh"\n#include <cstdio>\nint main() {\n' + "".join(
        "    {\n        const int d[] = {%s};\n        std::vector<int> off(1, 7);\n"
        "        for (int v : d) off.push_back(off.back() + v);\n"
        '        printf("%%d\\n", acs::host::soc_lanes(%d, off.data()));\n    }\n' % (", ".join(map(str, dims)), len(dims))
        for dims, _ in CASES) + '    printf("%d\\n", acs::host::soc_lanes(0, nullptr));\n}\n')
    exe = tmp_path / "lanes"
    subprocess.run([nvcc, "-std=c++17", f"-I{build.CSRC}", f"-I{build.INCLUDE}", "-o", str(exe), str(src)], check=True,
                   capture_output=True)
    got = [int(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
    assert got == [lanes for _, lanes in CASES] + [32]

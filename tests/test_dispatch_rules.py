"""Rules that choose between two forms of a step (csrc/launch.h), compiled as host code and
checked on the CPU at the sizes on both sides of their lines."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_01928_gb300", "csrc")


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    """rule("expression"): its value as an integer."""
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("rules")

    def value(expr):
        src, exe = d / "h.cu", d / "h"
        src.write_text('#include <cstdio>\n#include "launch.h"\nusing namespace debyefit;\n'
                       f'int main() {{ std::printf("%d", (int)({expr})); }}\n')
        r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src),
                            "-o", str(exe)], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-2000:]
        return int(subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout)
    return value


@pytest.mark.parametrize("longest,merged", [(0, 1), (1, 1), (4096, 1), (4097, 0), (1 << 30, 0)])
def test_preparation_goes_by_the_longest_spectrum(rule, longest, merged):
    assert rule(f"prep_merged({longest}ll)") == merged

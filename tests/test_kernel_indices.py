"""Index arithmetic that kernels share with the host, over its whole range, compiled for the host (no GPU)."""
import subprocess

import pytest

from paper_0707_1581_gb300 import build as B


def run_host(tmp_path, body: str, include: str) -> str:
    """Compiles a program of the library's own functions and returns what it prints."""
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(f'#include "{include}"\n#include <cstdio>\n#include <cstdlib>\nusing namespace flb;\n'
                   f"int main() {{\n{body}\n    return 0;\n}}\n")
    cmd = [B.nvcc(), *B.ARCH, "-std=c++17", "-O1", f"-I{B.INCLUDE}", f"-I{B.CSRC}", str(src), "-o", str(exe)]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, res.stdout + res.stderr
    return res.stdout


@pytest.mark.parametrize("units", [1, 5, 2 ** 27 - 1, 2 ** 27, 2 ** 27 + 100, 2 ** 31 - 1])
def test_every_unit_has_its_own_warp_of_the_plane_means(tmp_path, units):
    """Block b of 128 threads holds the units 4 b .. 4 b + 3, to the largest number of units a box can have."""
    run_host(tmp_path, f"""
    const long long units = {units}, blocks = (units + 3) / 4;
    for (long long b : {{0ll, 1ll, blocks / 2, blocks - 1}})
        for (unsigned t = 0; t < 128; ++t) {{
            const long long u = 4 * b + t / 32;
            if (b < blocks && u < units && profile::unit_of((unsigned)b, 128, t) != u) {{
                printf("block %lld thread %u: unit %d\\n", b, t, profile::unit_of((unsigned)b, 128, t));
                return 1;
            }}
        }}""", "profile.cuh")

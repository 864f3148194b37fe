"""CPU checks of what the kernels' header (csrc/fd_internal.h) shares with the host,
compiled as plain C++: row offsets past 2^31 cells, launch limits per device."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2403_17518_gb300", "csrc")


def run_host(tmp_path, body):
    """Output words of a C++ main() with `body` that includes the kernels' header."""
    cxx = shutil.which("g++")
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if cxx is None or not os.path.exists(nvcc):
        pytest.skip("no host compiler or CUDA headers")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    src = tmp_path / "host.cpp"
    src.write_text('#include <cstdio>\n#include "fd_internal.h"\nusing namespace dhfwi;\nint main() {\n' + body + "\n}\n")
    exe = tmp_path / "host"
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, "-I", cuda, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


def test_model_rows_of_large_models(tmp_path):
    cases = [(z, NZ, pf) for NZ, pf in ((141, 544), (4096, 524320), (3250, 700064), (65535, 32800))
             for z in (-4, 0, 1, NZ // 2, NZ - 1, NZ + 3)]
    body = "\n".join(f'std::printf("%lld\\n", (long long)model_row({z}, {NZ}, {pf}));' for z, NZ, pf in cases)
    got = [int(x) for x in run_host(tmp_path, body)]
    assert got == [min(max(z, 0), NZ - 1) * pf for z, NZ, pf in cases]
    assert max(got) >= 2**31


def test_launch_limits_belong_to_a_device(tmp_path):
    """Each device takes its own count, once; a device past the table takes it every time."""
    body = """
    static PerDevice p;
    int taken = 0;
    const int dev[] = {0, 1, 0, 63, 1, 64, 64};
    for (int d : dev) std::printf("%d ", p.get(d, [&] { taken++; return 100 + d; }));
    std::printf("%d", taken);"""
    assert [int(x) for x in run_host(tmp_path, body)] == [100, 101, 100, 163, 101, 164, 164, 5]

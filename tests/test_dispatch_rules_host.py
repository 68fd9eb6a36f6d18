"""The host's rules for routes and launches (csrc/tbs_internal.h), compiled by
nvcc into a small host program: no GPU needed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_13754_gb300", "csrc")


def _run(tmp_path, body):
    nvcc = next((c for c in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc") if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "harness.cu", tmp_path / "harness"
    src.write_text('#include <cstdio>\n#include "tbs_internal.h"\nusing namespace tbs;\nint main() {\n%s\nreturn 0;\n}\n'
                   % body)
    r = subprocess.run([nvcc, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()


def test_kernels_get_their_own_device_memory_only(tmp_path):
    """Host memory and another device's memory take the copies."""
    got = _run(tmp_path, r'''
    const cudaMemoryType t[4] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice,
                                 cudaMemoryTypeManaged};
    for (int k = 0; k < 4; k++)
        for (int m = 0; m < 2; m++) printf("%d ", (int)kernel_reaches(t[k], m, 1));
    ''')
    assert got == list("00000111")

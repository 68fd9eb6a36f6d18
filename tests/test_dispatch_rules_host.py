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


def test_graph_loops_launch_little_beyond_a_series(tmp_path):
    """Terms launched for a series of T terms.  To a residual: at most 6 within
    4, at most 7 beyond T, none beyond max_terms up to 12.  A fixed number: no
    body of at most 16 has fewer iterations (7 us) and empty terms (4 us)."""
    v = iter(_run(tmp_path, r'''
    for (int m = 1; m <= 300; m++)
        for (int r = 0; r < 2; r++) {
            const TermLoop l = term_loop(m, r != 0);
            printf("%d %d ", l.lead, l.body);
        }
    '''))
    for m in range(1, 301):
        for residual in (False, True):
            lead, body = int(next(v)), int(next(v))
            assert lead <= m and (lead == m) == (body == 0)

            def launched(t):
                return lead + (-(-max(t - lead, 0) // body) * body if body else 0)

            if residual:
                assert lead <= 6 and all(t <= launched(t) <= t + 7 for t in range(1, m + 1))
                assert m > 12 or launched(m) == m
            else:
                cost = [7 * -(-m // b) + 4 * (-(-m // b) * b - m) for b in range(1, min(m, 16) + 1)]
                assert lead == 0 and 7 * (launched(m) // body) + 4 * (launched(m) - m) == min(cost)


def test_reverse_loops_launch_few_empty_steps(tmp_path):
    """A sweep of S steps: none launched beyond max_terms - 1 up to 6 of them,
    at most 3 empty ones in a loop."""
    v = iter(_run(tmp_path, r'''
    for (int m = 1; m <= 300; m++) {
        const ReverseLoop l = reverse_loop(m);
        printf("%d %d ", l.lead, l.body);
    }
    '''))
    for m in range(1, 301):
        lead, body = int(next(v)), int(next(v))
        if m <= 7:
            assert (lead, body) == (m - 1, 0)
        else:
            assert lead == 0 and 3 <= body <= 4
            assert -(-(m - 1) // body) == -(-(m - 1) // 4)  # as few iterations as bodies of 4

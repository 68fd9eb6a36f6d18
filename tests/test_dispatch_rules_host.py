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


def test_synthesis_records_in_every_form():
    """The packed records are those of one structure per entry, for entries
    given in part, numbers of other types and refusals alike."""
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available to build the library")
    import ctypes
    import numpy as np
    from paper_2507_13754_gb300 import build, tbs
    build.build()
    f = tbs.tbs_synth_freq
    ok = [(0x1000, 8, 1e-4, 1e6, 1.0), (ctypes.c_void_p(0x2000), 8, 1e-4, 1e6, 1.0), (None, 9, 1, 2, 3),
          (0x3000, 2 ** 31 + 5, 0.5, -1e300, float("inf")), (0x4000, 8, np.float32(0.1), np.float64(3), True),
          (0x5000, 8), (0x6000, 8, 1e-4), ()]
    for entries in [[e] for e in ok] + [ok, ok[:1], []]:
        want = (f * len(entries))(*[f(*e) for e in entries])
        assert bytes(tbs._synth_records(entries)) == bytes(want)
    bad = [(0x1000, 8, "1e-4", 1e6, 1.0), (0x1000, 8.0, 1e-4, 1e6, 1.0), (0x1000, 8, 1e-4, 1e6, 1.0, 2.0)]
    for entries in [[e] for e in bad] + [[ok[0], bad[0]], [(0x1000, 8, 1e-4, 1e6), bad[2]]]:
        with pytest.raises(TypeError):
            [f(*e) for e in entries]
        with pytest.raises(TypeError):
            tbs._synth_records(entries)
    # synthesize() converts its numbers: text too
    text = tbs._synth_records([(0x1000, 8, "1e-4", "1e6", "0.5")], float)
    assert bytes(text) == bytes((f * 1)(f(0x1000, 8, 1e-4, 1e6, 0.5)))
    # short records reach the library's own checks (n_t = 0 is refused before any launch)
    with pytest.raises(tbs.TbsError):
        tbs.tbs_synthesize([(0x1000, 8)], 1, 0.0, 0.0, 1e-4, 1e-4, 1, 1, 0.0, 1e-8, 0, 0x2000)

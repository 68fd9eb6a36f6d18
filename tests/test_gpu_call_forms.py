"""Calls at the edges of what the entry points accept, and results that may
not depend on how a call is launched."""
import numpy as np
import pytest

from _helpers import gpu_plan, library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    library()


@pytest.mark.parametrize("off_c,off_a", [(1, 0), (0, 2), (3, 1)])
def test_medium_at_any_address(off_c, off_a):
    """c and alpha packed in a byte buffer, off a float's boundary: the field
    is that of aligned ones, bit for bit."""
    import torch
    from paper_2507_13754_gb300 import tbs, workloads as W
    w = W.random_medium(40, seed=70, n_rhs=2)

    def packed(a, off):
        raw = torch.zeros(a.nbytes + 4, dtype=torch.uint8, device="cuda")
        raw[off:off + a.nbytes] = torch.from_numpy(a.view(np.uint8).ravel()).cuda()
        return raw, raw.data_ptr() + off

    out = []
    for oc, oa in ((0, 0), (off_c, off_a)):
        p = gpu_plan(w, max_terms=6, tol=0.0)
        (cb, cp), (ab, ap) = packed(w.c, oc), packed(w.alpha, oa)
        tbs.tbs_set_medium(p.handle, cp, ap, w.ypow, w.f_ref, torch.cuda.current_stream().cuda_stream)
        p.set_sources(w.src_ix, w.src_iy, w.src_amp)
        out.append(p.solve()[0].cpu().numpy())
        p.close()
    assert np.abs(out[0]).max() > 0
    assert np.array_equal(out[0], out[1])

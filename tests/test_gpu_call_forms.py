"""Calls at the edges of what the entry points accept, and results that may
not depend on how a call is launched."""
import numpy as np
import pytest

from _helpers import gpu_plan, library, rel_l2

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


# 2e-7: the bar of the other spectrum tests (one rounding to complex64).  At
# k0 dx = 1e-27 the orders of the cell modes overflow FP64.
@pytest.mark.parametrize("kh", [1e-27, 1e-18, 0.9e-9, 1.1e-9])
@pytest.mark.parametrize("n", [9, 33])
def test_ghat_at_any_fine_sampling(oracle_mod, n, kh):
    import math
    from paper_2507_13754_gb300 import tbs
    c0, dx = 1500.0, 1e-3
    f = kh * c0 / (2 * math.pi * dx)
    plan = tbs.Plan(n, dx, f, c0)
    gh = oracle_mod.ghat(n, plan.m, dx, oracle_mod.green_table(n, 2 * math.pi * f / c0, dx))
    q = plan.m // 2 + 1
    assert rel_l2(plan.ghat_quadrant(), gh[:q, :q]) < 2e-7
    plan.close()

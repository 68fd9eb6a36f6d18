"""Edges of the kernels' size rules on the GPU: narrow and wide column tiles,
row blocks of 64 and 256 threads, the compact column pass, the persistent row
passes at odd N, the stop test inside the column pass, the outputs' small and
general routes, the synthesis's two phase reductions."""
import numpy as np
import pytest

from _helpers import PARITY_RTOL, gpu_solve, library, oracle_solve, rel_l2
from test_gpu_adjoint_harmonic import GRAD_RTOL, _gpu_forward, _oracle_gradient

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    library()


# M = 64 (separate stop kernel); 128 and 256 at the last narrow and first wide
# number of RHS; 512 around 64/256-thread row blocks (152 x 256 threads), odd N;
# 1024; 2048 (compact) at the ends of its range; 4096 at its smallest N
@pytest.mark.parametrize("n,n_rhs", [(17, 2), (33, 4), (64, 5), (65, 2), (128, 3), (129, 1), (255, 4), (256, 5),
                                     (257, 1), (511, 2), (513, 2), (1023, 1), (1024, 1), (1025, 1)])
def test_solve_matches_oracle_at_size_edges(n, n_rhs):
    from paper_2507_13754_gb300 import workloads as W
    w = W.random_medium(n, seed=61, n_rhs=n_rhs)
    w.max_terms, w.tol = 9, 0.0
    psi, info, plan = gpu_solve(w)
    assert [i["terms"] for i in info] == [9] * n_rhs
    for r, (ref, *_rest) in enumerate(oracle_solve(w)):
        assert rel_l2(psi[r], ref) < PARITY_RTOL, (n, r)
    plan.close()


@pytest.mark.parametrize("n,max_terms", [(96, 3), (96, 8), (96, 40), (257, 17), (300, 40)])
def test_graph_bodies_and_unrolled_launches_stop_alike(n, max_terms):
    """RHS that stop after different numbers of terms (one has no source at
    all), whatever the place of their last term in the graph's loop body."""
    from paper_2507_13754_gb300 import workloads as W
    w = W.random_medium(n, seed=62, n_rhs=4)
    w.src_amp[2] = 0
    w.src_amp[3] *= 1e-3
    w.max_terms, w.tol = max_terms, 1e-5
    psi0, info0, p0 = gpu_solve(w)
    psi1, info1, p1 = gpu_solve(w, use_graph=False)
    assert info0 == info1
    assert np.array_equal(psi0, psi1)
    for r, (ref, rinfo, *_rest) in enumerate(oracle_solve(w)):
        if np.any(w.src_amp[r]):
            assert abs(info0[r]["terms"] - rinfo["terms"]) <= 1
    p0.close()
    p1.close()


@pytest.mark.parametrize("n,n_rhs", [(257, 1), (301, 2), (512, 1), (513, 1)])
def test_reverse_sweep_at_odd_and_even_n(n, n_rhs):
    """Also more than one iteration of the reverse loop (8 steps each)."""
    import torch
    from paper_2507_13754_gb300 import workloads as W
    w = W.random_medium(n, seed=63, n_rhs=n_rhs)
    plan, psi, info = _gpu_forward(w, max_terms=12, tol=0.0)
    rng = np.random.default_rng(163)
    g = (rng.standard_normal((n_rhs, n, n)) + 1j * rng.standard_normal((n_rhs, n, n))).astype(np.complex64)
    gc = torch.empty((n, n), dtype=torch.float32, device="cuda")
    ga = torch.empty((n, n), dtype=torch.float32, device="cuda")
    plan.solve_adjoint(torch.from_numpy(g).cuda(), gc, ga)
    rc, ra = _oracle_gradient(w, [i["terms"] for i in info], g)
    assert rel_l2(gc.cpu().numpy(), rc) < GRAD_RTOL
    assert rel_l2(ga.cpu().numpy(), ra) < GRAD_RTOL
    plan.close()


@pytest.mark.parametrize("n,ks", [(256, False), (256, True), (512, False), (512, True), (1024, False), (1024, True)])
def test_periodic_tiles_give_one_result(n, ks):
    """One RHS (narrow tiles) and the same RHS among four (wide or compact
    tiles): the same arithmetic, bit for bit."""
    import math
    import torch
    from paper_2507_13754_gb300 import tbs, workloads as W
    w = W.random_medium(n, seed=64, n_rhs=4)
    k0 = 2 * math.pi * w.f / w.c0
    kw = dict(kspace_alpha0=2e-8, kspace_nu=1.5) if ks else {}
    out = []
    for rhs in (1, 4):
        p = tbs.Plan(n, w.dx, w.f, w.c0, n_rhs=rhs, max_terms=10, tol=0.0, periodic=True, abl_width=16,
                     abl_zeta=4.0 / (16 * w.dx), div_window=1 << 30, div_factor=math.inf, **kw)
        p.set_potential(torch.full((n, n), 0.0 if ks else 0.05 * k0 * k0, dtype=torch.complex64, device="cuda"))
        p.set_sources(w.src_ix, w.src_iy, w.src_amp[:rhs])
        out.append(p.solve()[0].cpu().numpy())
        p.close()
    assert np.abs(out[0]).max() > 0
    assert np.array_equal(out[0][0], out[1][0])


def test_outputs_at_any_alignment():
    """Fields that start 8 bytes past a 16-byte boundary and records at an odd
    address take the general copies; the results are those of aligned ones."""
    import ctypes
    import torch
    from paper_2507_13754_gb300 import tbs, workloads as W
    w = W.random_medium(64, seed=65, n_rhs=2)
    psi0, info0, plan = gpu_solve(w)
    need = 2 * ctypes.sizeof(tbs.tbs_solve_info)
    psi = torch.zeros(2 * 64 * 64 + 1, dtype=torch.complex64, device="cuda")[1:].view(2, 64, 64)
    raw = torch.zeros(need + 1, dtype=torch.uint8, device="cuda")
    plan.solve(psi=psi, info=raw[1:])
    assert np.array_equal(psi.cpu().numpy(), psi0)
    assert plan.device_info_dicts(raw[1:].clone()) == info0
    plan.close()


@pytest.mark.parametrize("t0,nt", [(1e-4, 255), (1e-4, 257), (3e-2, 257)])
def test_synthesis_phase_reductions(t0, nt):
    """|f t| below 2^16 cycles (FP32 pairs) and above (FP64), 17 receivers
    (one past a block's), either side of a block's 256 times.  The bound is
    that of the other synthesis tests."""
    import torch
    import oracle
    from paper_2507_13754_gb300 import tbs
    rng = np.random.default_rng(66)
    ns, freqs, w = [8, 13, 21], [2.1e6, 3.7e6, 5.3e6], [0.5, 1.0, 0.7]
    dxs = [6e-3 / n for n in ns]
    fields = [(rng.standard_normal((2, n, n)) + 1j * rng.standard_normal((2, n, n))).astype(np.complex64) for n in ns]
    args = (dxs, freqs, w, (0.1e-3, 1e-3), (0.3e-3, 0.0), (17, 1), t0, 1.1e-8, nt)
    s = tbs.synthesize([torch.from_numpy(f).cuda() for f in fields], *args).cpu().numpy()
    ref = oracle.synthesize([f.astype(np.complex128) for f in fields], *args)
    assert rel_l2(s, ref) < PARITY_RTOL

"""Calls at the edges of what the entry points accept, and results that may
not depend on how a call is launched."""
import numpy as np
import pytest

from _helpers import gpu_plan, gpu_solve, library, rel_l2

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


def _phases(f, t0, dt, nt):
    """exp(-2 pi i f t_j): the signal of a field of ones at weight 1."""
    import torch
    from paper_2507_13754_gb300 import tbs
    ones = torch.ones((1, 2, 2), dtype=torch.complex64, device="cuda")
    return tbs.synthesize([ones], [1.0], [f], [1.0], (0.0, 0.0), (0.0, 0.0), (1, 1), t0, dt, nt).cpu().numpy().ravel()


# a phase rounded to FP32 (1.5e-8 cycles, 9.4e-8 rad) and the two components'
# rounding (one unit in the last place each, 8.5e-8 together)
@pytest.mark.parametrize("f,t0,dt,nt", [(1e39, 0.0, 0.0, 1), (-1e300, 0.0, 0.0, 3), (2.5e31, 1e-31, 1e-32, 5)])
def test_synthesis_at_frequencies_beyond_fp32(f, t0, dt, nt):
    t = t0 + np.arange(nt) * dt
    assert np.abs(_phases(f, t0, dt, nt) - np.exp(-2j * np.pi * (f * t - np.rint(f * t)))).max() < 1.8e-7


# |f t| to 2^16 cycles: the phase within 6e-10 cycles (4e-9 rad), sine and
# cosine to one unit in the last place and one more rounding (9e-8 each)
@pytest.mark.parametrize("f", [3.7, 5.123456e6])
def test_synthesis_phase_error(f):
    nt = 1 << 20
    dt = 64729.13579 / f / nt
    cyc = np.longdouble(f) * (np.arange(nt) * dt).astype(np.longdouble)
    ref = np.exp(-2j * np.pi * (cyc - np.rint(cyc)).astype(np.float64))
    assert np.abs(_phases(f, 0.0, dt, nt) - ref).max() < 1.33e-7


@pytest.mark.parametrize("n", [257, 511, 513, 1025])
def test_norms_of_odd_grids(n):
    """psi_norm against FP64 sums of each thread's FP32 sum of squares (formed
    here from the field it belongs to): the sums across threads carry double-
    float pairs, 48 bits.  1e-10 leaves room for a thread's sum that this
    emulation rounds twice (6e-8 of one of n^2 / 8 sums)."""
    from paper_2507_13754_gb300 import workloads as W
    w = W.random_medium(n, seed=72)
    w.max_terms, w.tol = 4, 0.0
    psi, info, plan = gpu_solve(w)
    T = plan.m // 16
    x = np.zeros((n, 8 * T, 2))
    x[:, :n, 0], x[:, :n, 1] = psi[0].real, psi[0].imag
    x = x.reshape(n, 8, T, 2)
    s = np.zeros((n, T), np.float32)
    for m in range(8):
        s = (x[:, m, :, 1] ** 2 + s).astype(np.float32)
        s = (x[:, m, :, 0] ** 2 + s).astype(np.float32)
    assert abs(info[0]["psi_norm"] / np.sqrt(s.sum(dtype=np.float64)) - 1) < 1e-10
    plan.close()


@pytest.mark.parametrize("n,n_rhs", [(64, 16), (128, 24), (256, 24), (512, 8), (1024, 8)])
def test_records_do_not_depend_on_the_launch(n, n_rhs):
    """The same bits whether a term's stop test is made by a kernel of its own
    (the last of max_terms, launched from the host), inside a column pass of
    any tile shape (a term that ends a series to a residual), with the RHS
    alone in its plan or among others.  The periodic grid's Green's function
    decays: the rows' sums span so many binades that another order of theirs
    rounds otherwise."""
    import math
    import torch
    from paper_2507_13754_gb300 import tbs, workloads as W
    w = W.random_medium(n, seed=71, n_rhs=n_rhs)
    k0 = 2 * math.pi * w.f / w.c0

    def solve(amp, max_terms, tol, variant=0, **kw):
        p = tbs.Plan(n, w.dx, w.f, w.c0, n_rhs=len(amp), max_terms=max_terms, tol=tol, periodic=True,
                     div_window=1 << 30, div_factor=math.inf, **kw)
        p.set_potential(torch.full((n, n), 0.05 * k0 * k0, dtype=torch.complex64, device="cuda"))
        p.set_sources(w.src_ix, w.src_iy, amp)
        variants = tbs.tbs_col_variants(p.handle)
        tbs.tbs_set_col_variant(p.handle, variant % variants)
        info = tbs.Plan.info_dicts(p.solve()[1])
        p.close()
        return [(i["terms"], i["residual"], i["term_norm_max"], i["psi_norm"]) for i in info], variants

    ref, variants = solve(w.src_amp, 3, 0.0, use_graph=False)
    tol = max(r[1] for r in ref) * (1 + 1e-6)
    assert all(r[0] == 3 for r in ref) and 0 < tol < 1
    for v in range(variants):
        got, _ = solve(w.src_amp, 40, tol, v)
        ended = [r for r in range(n_rhs) if got[r][0] == 3]
        assert ended
        assert [got[r] for r in ended] == [ref[r] for r in ended], v
    for r in range(0, n_rhs, 3):
        one, _ = solve(w.src_amp[r:r + 1], 40, ref[r][1] * (1 + 1e-6))
        assert one[0] == ref[r], r


@pytest.mark.parametrize("n,n_rhs", [(20, 700), (64, 300), (140, 70), (260, 40)])
def test_many_rhs_stop_on_their_own(n, n_rhs):
    """Hundreds of RHS that stop after different numbers of terms: each has the
    field and records that it has in a plan of its own few."""
    from paper_2507_13754_gb300 import workloads as W
    w = W.random_medium(n, seed=73, n_rhs=n_rhs)
    w.alpha *= np.float32(1500.0 / n)
    w.src_amp[::3, 1:] = 0
    w.src_amp[5] = 0
    psi, info, plan = gpu_solve(w, max_terms=40, tol=1e-4)
    plan.close()
    assert len({i["terms"] for i in info}) > 1
    amp = w.src_amp
    for r0 in range(0, n_rhs, 9):
        w.src_amp = amp[r0:r0 + 5]
        some, some_info, p = gpu_solve(w, max_terms=40, tol=1e-4)
        assert some_info == info[r0:r0 + 5]
        assert np.array_equal(some, psi[r0:r0 + 5])
        p.close()


@pytest.mark.parametrize("n", [258, 512, 700])
def test_reverse_sweep_is_the_same_for_both_row_variants(n):
    """The row variants are the forward pass's: the gradients agree bit for bit."""
    import torch
    from paper_2507_13754_gb300 import tbs, workloads as W
    w = W.random_medium(n, seed=74, n_rhs=2)
    rng = np.random.default_rng(174)
    g = torch.from_numpy((rng.standard_normal((2, n, n)) + 1j * rng.standard_normal((2, n, n))).astype(np.complex64))
    _, _, plan = gpu_solve(w, keep_terms=True, max_terms=9, tol=0.0)
    out = []
    for v in (0, 1):
        tbs.tbs_set_row_variant(plan.handle, v)
        plan.solve()
        gc = torch.empty((n, n), dtype=torch.float32, device="cuda")
        ga = torch.empty((n, n), dtype=torch.float32, device="cuda")
        plan.solve_adjoint(g.cuda(), gc, ga)
        out.append((gc.cpu().numpy(), ga.cpu().numpy()))
    plan.close()
    assert np.abs(out[0][0]).max() > 0
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("n,max_terms", [(257, 30), (300, 20), (513, 12)])
def test_checkpointed_sweep_of_persistent_passes(n, max_terms):
    """M >= 512: the reverse pass bulk-copies the recomputed terms of a segment
    (odd rows 8 bytes off a 16-byte boundary): bitwise the stored sweep, for RHS
    with different term counts over several segments."""
    import torch
    from paper_2507_13754_gb300 import tbs, workloads as W
    w = W.random_medium(n, seed=75, n_rhs=3)
    w.src_amp[1] *= 0.5
    w.src_amp[2] = 0
    rng = np.random.default_rng(175)
    g = (rng.standard_normal((3, n, n)) + 1j * rng.standard_normal((3, n, n))).astype(np.complex64)
    out = []
    for ck in (False, True):
        psi, info, plan = gpu_solve(w, keep_terms=True, checkpoint=ck, max_terms=max_terms, tol=1e-12)
        gc = torch.empty((n, n), dtype=torch.float32, device="cuda")
        ga = torch.empty((n, n), dtype=torch.float32, device="cuda")
        plan.solve_adjoint(torch.from_numpy(g).cuda(), gc, ga)
        out.append((info, psi, gc.cpu().numpy(), ga.cpu().numpy()))
        plan.close()
    (i0, p0, c0, a0), (i1, p1, c1, a1) = out
    assert i0 == i1 and i0[2]["terms"] == 1 and max(i["terms"] for i in i0) > 8
    assert np.abs(c0).max() > 0 and np.array_equal(p0, p1)
    assert np.array_equal(c0, c1) and np.array_equal(a0, a1)


@pytest.mark.parametrize("n,n_rhs,narrow", [(64, 1, True), (64, 4, True), (64, 5, False), (128, 2, True),
                                            (128, 3, False), (32, 1, False)])
def test_variant_names_tell_narrowed_tiles(n, n_rhs, narrow):
    from paper_2507_13754_gb300 import tbs
    p = tbs.Plan(n, 1e-4, 1e6, 1500.0, n_rhs=n_rhs)
    name = tbs.tbs_col_variant_name(p.handle)
    assert ("narrowed" in name) == narrow and ("default width" in name) == (not narrow)
    p.close()


def test_a_series_that_ends_costs_no_column_pass():
    """The column pass under way when the last series ends is broken off: two
    terms to a residual take less than three quarters of a column pass more than
    two terms that nothing follows (least of many runs)."""
    import torch
    from paper_2507_13754_gb300 import workloads as W

    def least(plan):
        psi, _ = plan.solve()
        info = torch.empty(64 * plan.n_rhs, dtype=torch.uint8, device="cuda")
        ms = []
        for _ in range(40):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            plan.solve(psi=psi, info=info, sync=False)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms)

    w = W.random_medium(1024, seed=76, n_rhs=8)
    w.alpha *= np.float32(0.05)  # weak enough for the second term to be the smaller one
    w.c[:] = 1500 + (w.c - 1500) * np.float32(0.1)
    _, info, two = gpu_solve(w, max_terms=2, tol=0.0)
    _, to_tol, series = gpu_solve(w, max_terms=64, tol=max(i["residual"] for i in info) * (1 + 1e-6))
    assert [i["terms"] for i in to_tol] == [2] * 8
    extra = least(series) - least(two)
    two.set_timing()
    two.solve()
    _, _, col_ms, cols = two.timing()
    assert extra < 0.75 * col_ms / cols, (extra, col_ms / cols)
    two.close()
    series.close()

"""The Green's table over the samplings a plan accepts: direct quadrature near
the origin, cell modes beyond (one or two fitted intervals per cell of r), the
6 x 6 rule above k0 dx = 2, and grids at the near square's edge."""
import math

import numpy as np
import pytest

from _helpers import library, rel_l2

pytestmark = pytest.mark.gpu


# The table is formed in FP64 and its spectrum rounded once to complex64
# (2^-24 = 6e-8 per entry): the bar of the other spectrum test, 2e-7.
@pytest.mark.parametrize("n", [7, 8, 9, 10, 33, 65, 200])
@pytest.mark.parametrize("kh", [1e-3, 0.4, 1.0, 1.01, math.pi / 2, 2.0, 2.01])
def test_ghat_over_samplings(oracle_mod, n, kh):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    library()
    from paper_2507_13754_gb300 import tbs
    c0, f = 1500.0, 1e6
    k0 = 2 * math.pi * f / c0
    dx = kh / k0
    plan = tbs.Plan(n, dx, f, c0)
    gh = oracle_mod.ghat(n, plan.m, dx, oracle_mod.green_table(n, k0, dx))
    q = plan.m // 2 + 1
    assert rel_l2(plan.ghat_quadrant(), gh[:q, :q]) < 2e-7
    plan.close()

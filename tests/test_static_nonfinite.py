"""Non-finite populations: the static step without the flux terms gives what the
one with them gives (a lambda field of zeros takes the latter)."""
import numpy as np
import pytest

from paper_2007_05718_gb300 import lbrt
from paper_2007_05718_gb300 import workloads as W

pytestmark = pytest.mark.gpu
ICO = [dict(dirset=lbrt.LB_RT_ICOSPHERE, level=l) for l in (0, 1, 2)]


@pytest.mark.parametrize("storage", [lbrt.LB_RT_F32, lbrt.LB_RT_F16_DEV, lbrt.LB_RT_BF16_DEV])
@pytest.mark.parametrize("collision", [lbrt.LB_RT_IMPLICIT_EXACT, lbrt.LB_RT_EXPLICIT, lbrt.LB_RT_LAMBDA_K])
@pytest.mark.parametrize("level", [0, 1, 2])
def test_flux_terms_of_non_finite_populations(cuda, storage, collision, level):
    shape = (9, 5, 66)
    N = 10 * 4 ** level + 2
    S = W.random_populations(N, shape, 5)
    for k, v in enumerate((np.inf, np.nan, -np.inf, np.inf)):
        S[(11 * k) % N, 2 * k, k, 16 * k + 3] = v
    got = []
    for lam in (0.0, np.zeros(shape, np.float32)):
        h = lbrt.lb_rt_create(3, 66, 5, 9, storage=storage, collision=collision, lambda_iters=2, **ICO[level])
        try:
            lbrt.lb_rt_set_fluid(h, kappa_a=1.0, kappa_0=2.0, lam=lam, eta=1.0)
            lbrt.lb_rt_set_state(h, S)
            for _ in range(2):
                lbrt.lb_rt_step(h, 1)
                got.append(np.zeros((N,) + shape, np.float32))
                lbrt.lb_rt_get_populations(h, got[-1])
        finally:
            lbrt.lb_rt_destroy(h)
    assert not np.isfinite(got[0]).all() and np.isfinite(got[0]).any()
    assert np.array_equal(got[0], got[2], equal_nan=True)
    assert np.array_equal(got[1], got[3], equal_nan=True)

"""Moments and coupling outputs, two sites a thread and (with P, or from 96
directions on) eight directions at a time: remainders of the directions, odd rows."""
import numpy as np
import pytest

from paper_2007_05718_gb300 import lbrt
from paper_2007_05718_gb300 import workloads as W

pytestmark = pytest.mark.gpu
ICO = [dict(dirset=lbrt.LB_RT_ICOSPHERE, level=l) for l in (0, 1, 2)]
GL = lambda a, b: dict(dirset=lbrt.LB_RT_GAUSS_LEGENDRE, gl=(a, b))  # noqa: E731
DIRS = [dict(dirs=[[0.0, 0.0, 1.0]]), dict(dirs=np.eye(3)), ICO[0], ICO[1], ICO[2], GL(6, 12), GL(8, 12), GL(11, 9)]


@pytest.mark.parametrize("storage", [lbrt.LB_RT_F32, lbrt.LB_RT_F16_DEV, lbrt.LB_RT_BF16_DEV])
@pytest.mark.parametrize("dirs", DIRS, ids=["1", "3", "12", "42", "162", "72", "96", "99"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 7), (2, 3, 64), (5, 2, 33)], ids=str)
def test_moments_and_coupling_of_the_stored_populations(cuda, storage, dirs, shape):
    nz, ny, nx = shape
    h = lbrt.lb_rt_create(3, nx, ny, nz, storage=storage, collision=lbrt.LB_RT_EXPLICIT, **dirs)
    try:
        n = lbrt.lb_rt_directions(h)[0]
        N = len(n)
        lbrt.lb_rt_set_fluid(h, kappa_a=0.5, kappa_0=2.0, eta=0.25)
        lbrt.lb_rt_set_state(h, W.random_populations(N, shape, 7))
        I = np.zeros((N,) + shape, np.float32)
        lbrt.lb_rt_get_populations(h, I)
        E, F, Pt = (np.zeros(s + shape, np.float32) for s in ((), (3,), (6,)))
        E2, F2 = np.zeros_like(E), np.zeros_like(F)
        J, H, S = (np.zeros(s + shape, np.float32) for s in ((), (3,), (4,)))
        lbrt.lb_rt_moments(h, E, F, Pt)
        lbrt.lb_rt_moments(h, E2, F2)
        lbrt.lb_rt_coupling(h, J, H, S)
    finally:
        lbrt.lb_rt_destroy(h)
    I, n = I.astype(np.float64), np.asarray(n, np.float64)
    e = I.sum(0)
    f = np.einsum("ia,izyx->azyx", n, I)
    p = np.stack([np.einsum("i,i,izyx->zyx", n[:, a], n[:, b], I)
                  for a, b in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))])
    tol = (N + 8) * 2.0 ** -23 * e.max()  # N float32 additions, a few roundings of n, n n and w E^ (1 + q)
    for got, want in ((E, e), (F, f), (Pt, p), (J, e), (H, f)):
        assert np.abs(got - want).max() <= tol
    assert np.array_equal(E, E2) and np.array_equal(F, F2)
    four = np.concatenate([(0.5 * e - 0.25)[None], 2.5 * f])  # at rest: kt_a J - eta_t, kt H
    assert np.abs(S - four).max() <= 4 * tol

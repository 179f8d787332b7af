"""Energy budget of the static step: a partial sum per tile, whichever CTA ran
the tile."""
import numpy as np
import pytest

from paper_2007_05718_gb300 import lbrt
from paper_2007_05718_gb300 import workloads as W

pytestmark = pytest.mark.gpu
P, V = lbrt.LB_RT_PERIODIC, lbrt.LB_RT_VACUUM
ICO = [dict(dirset=lbrt.LB_RT_ICOSPHERE, level=l) for l in (0, 1, 2)]
RING = lambda n: dict(dirset=lbrt.LB_RT_RING2D, ndir=n)  # noqa: E731
# total is sum E' in float64 of float32 collision scalars, E the sum over the
# stored populations (uniform in [0, 1) / N, so |q| < 1 in 16 bits): per site
# they differ by N float32 roundings, or by one of q
BOUND = {lbrt.LB_RT_F32: 162 * 2.0 ** -23, lbrt.LB_RT_F16_DEV: 2.0 ** -11, lbrt.LB_RT_BF16_DEV: 2.0 ** -8}


@pytest.mark.parametrize("dims,shape,dirs,bc", [
    (3, (40, 61, 70), ICO[1], (P, P, P)),     # more tiles than CTAs
    (3, (1, 300, 64), ICO[1], (P, V, P)),     # tiles of one batch
    (3, (2, 1, 3), ICO[1], (V, V, V)),        # one tile
    (3, (37, 40, 130), ICO[2], (P, V, P)),
    (3, (5, 9, 33), ICO[0], (V, P, V)),
    (2, (1, 700, 200), RING(120), (P, V, P)),
    (2, (1, 64, 64), RING(16), (V, P, P)),
], ids=str)
@pytest.mark.parametrize("storage", [lbrt.LB_RT_F32, lbrt.LB_RT_F16_DEV, lbrt.LB_RT_BF16_DEV])
@pytest.mark.parametrize("lam", [0.0, 0.3])
def test_budget_sums_every_tile_in_one_order(cuda, dims, shape, dirs, bc, storage, lam):
    nz, ny, nx = shape
    h = lbrt.lb_rt_create(dims, nx, ny, nz, storage=storage, bc=bc, budget=True, **dirs)
    try:
        N = lbrt.lb_rt_directions(h)[0].shape[0]
        lbrt.lb_rt_set_fluid(h, kappa_a=1.0, kappa_0=5.0, lam=lam, eta=W.random_fields(shape, 2, 0.0, 2.0))
        I0 = W.random_populations(N, shape, 3)
        runs = []
        for _ in range(2):
            lbrt.lb_rt_set_state(h, I0)
            lbrt.lb_rt_step(h, 3)
            E = np.zeros(shape, np.float32)
            runs.append(lbrt.lb_rt_moments(h, E, budget=True))
    finally:
        lbrt.lb_rt_destroy(h)
    assert runs[0] == runs[1]
    b, total = runs[0], E.sum(dtype=np.float64)
    assert b["steps"] == 3
    assert abs(b["total"] - total) <= BOUND[storage] * total
    assert abs(b["total"] - b["initial"] - b["source"] + b["outflow"] - b["injection"]) <= 1e-12 * total

"""Every route of the static step gives the same bits: with and without the flux
terms (a lambda field of zeros takes the kernel that has them), tiles taken from
the counter or dealt out in advance (the energy budget), one problem or a batch;
at the edges of tiles, rows, planes and direction plans."""
import numpy as np
import pytest

from paper_2007_05718_gb300 import lbrt
from paper_2007_05718_gb300 import workloads as W

pytestmark = pytest.mark.gpu
P, V = lbrt.LB_RT_PERIODIC, lbrt.LB_RT_VACUUM
F32, F16, BF16 = lbrt.LB_RT_F32, lbrt.LB_RT_F16_DEV, lbrt.LB_RT_BF16_DEV
STEPS = 5


def _run(dims, shape, dirset, storage, bc, lam_field, budget=False):
    nz, ny, nx = shape
    h = lbrt.lb_rt_create(dims, nx, ny, nz, storage=storage, bc=bc, budget=budget, **dirset)
    try:
        N = lbrt.lb_rt_directions(h)[0].shape[0]
        lam = np.zeros(shape, np.float32) if lam_field else 0.0
        lbrt.lb_rt_set_fluid(h, kappa_a=W.random_fields(shape, 1, 0.0, 5.0), kappa_0=3.0, lam=lam,
                             eta=W.random_fields(shape, 2, 0.0, 2.0))
        lbrt.lb_rt_set_state(h, W.random_populations(N, shape, 3))
        lbrt.lb_rt_step(h, STEPS)
        I = np.zeros((N,) + shape, np.float32)
        lbrt.lb_rt_get_populations(h, I)
        return I
    finally:
        lbrt.lb_rt_destroy(h)


ICO = [dict(dirset=lbrt.LB_RT_ICOSPHERE, level=l) for l in (0, 1, 2)]
RING = lambda n: dict(dirset=lbrt.LB_RT_RING2D, ndir=n)  # noqa: E731
GL = lambda a, b: dict(dirset=lbrt.LB_RT_GAUSS_LEGENDRE, gl=(a, b))  # noqa: E731


@pytest.mark.parametrize("dims,shape,dirset,bc", [
    (3, (17, 5, 63), ICO[1], (P, P, P)), (3, (16, 3, 64), ICO[1], (P, V, P)),
    (3, (33, 2, 65), ICO[1], (V, P, V)), (3, (2, 1, 130), ICO[1], (P, P, P)),
    (3, (1, 7, 1), ICO[1], (P, P, P)), (3, (18, 4, 128), ICO[2], (P, P, P)),
    (3, (5, 3, 66), ICO[2], (V, V, V)), (3, (3, 2, 2), ICO[2], (P, P, V)),
    (3, (9, 5, 40), ICO[0], (P, V, V)), (3, (6, 5, 33), GL(4, 8), (P, P, V)),
    (3, (6, 5, 33), GL(6, 12), (V, P, P)), (3, (4, 3, 70), GL(8, 16), (P, P, P)),
    (2, (1, 1, 64), RING(16), (P, P, P)), (2, (1, 2, 65), RING(16), (V, P, P)),
    (2, (1, 41, 130), RING(120), (P, V, P)), (2, (1, 17, 63), RING(38), (P, P, P)),
    (2, (1, 300, 20), RING(8), (V, V, P)),
], ids=str)
@pytest.mark.parametrize("storage", [F32, F16, BF16])
def test_routes_of_the_static_step_agree(cuda, dims, shape, dirset, bc, storage):
    plain = _run(dims, shape, dirset, storage, bc, lam_field=False)
    assert np.isfinite(plain).all() and (plain > 0).any()
    flux = _run(dims, shape, dirset, storage, bc, lam_field=True)
    assert np.array_equal(plain, flux)
    dealt = _run(dims, shape, dirset, storage, bc, lam_field=False, budget=True)
    assert np.array_equal(plain, dealt)


@pytest.mark.parametrize("storage", [F32, F16])
@pytest.mark.parametrize("lam", [0.0, 0.4])
def test_batch_of_uneven_grids_agrees_with_single_problems(cuda, storage, lam):
    """2D and 3D problems, some with a lambda, in one batch."""
    probs = [(3, (9, 5, 63), ICO[1]), (3, (12, 3, 65), ICO[2]), (2, (1, 40, 66), RING(38)), (3, (2, 2, 3), ICO[1])]
    b = lbrt.lb_rt_batch_create(max_problems=8, storage=storage, steps_per_tick=STEPS, pair_groups=2)
    try:
        got = []
        for k, (dims, shape, dirset) in enumerate(probs):
            nz, ny, nx = shape
            E0 = W.random_fields(shape, 20 + k)
            slot = lbrt.lb_rt_batch_admit(b, dict(dims=dims, nx=nx, ny=ny, nz=nz, **dirset),
                                          dict(kappa_0=2.0, lam=lam if k % 2 == 0 else 0.0), E0,
                                          lbrt.LB_RT_STATE_ISOTROPIC, 4 * STEPS)
            got.append((slot, np.zeros(shape, np.float32), np.zeros((3,) + shape, np.float32)))
        for _ in range(4):
            lbrt.lb_rt_batch_tick(b)
        lbrt.lb_rt_batch_sync(b)
        for slot, E, F in got:
            lbrt.lb_rt_batch_moments(b, slot, E, F)
    finally:
        lbrt.lb_rt_batch_destroy(b)
    for k, ((dims, shape, dirset), (_, E, F)) in enumerate(zip(probs, got)):
        nz, ny, nx = shape
        h = lbrt.lb_rt_create(dims, nx, ny, nz, storage=storage, **dirset)
        try:
            lbrt.lb_rt_set_fluid(h, kappa_0=2.0, lam=lam if k % 2 == 0 else 0.0)
            lbrt.lb_rt_set_state(h, W.random_fields(shape, 20 + k), lbrt.LB_RT_STATE_ISOTROPIC)
            lbrt.lb_rt_step(h, 4 * STEPS)
            E1, F1 = np.zeros_like(E), np.zeros_like(F)
            lbrt.lb_rt_moments(h, E1, F1)
        finally:
            lbrt.lb_rt_destroy(h)
        assert np.array_equal(E, E1) and np.array_equal(F, F1)


@pytest.mark.parametrize("storage", [F32, F16])
@pytest.mark.parametrize("shape", [(1, 5, 63), (1, 17, 130)])
def test_saved_state_of_a_2d_grid_holds_the_z_mirrors(shape, storage):
    """The step leaves out the mirror planes of a 2D grid's periodic z axis; a
    saved state has them all the same: three equal planes per array."""
    nz, ny, nx = shape
    h = lbrt.lb_rt_create(2, nx, ny, nz, storage=storage, bc=(P, V, P), **RING(12))
    try:
        lbrt.lb_rt_set_fluid(h, kappa_a=2.0, eta=1.0)
        lbrt.lb_rt_set_state(h, W.random_populations(12, shape, 3))
        lbrt.lb_rt_step(h, 3)
        raw = np.frombuffer(lbrt.lb_rt_save_state(h), np.uint8)
    finally:
        lbrt.lb_rt_destroy(h)
    body = raw[64:-64]
    row = (nx + 3 + 7) // 8 * 8  # sites of a padded row
    e_bytes = 0 if storage == F32 else 3 * 4 * row * (ny + 2)
    for a in (body[:body.size - e_bytes], body[body.size - e_bytes:]):
        planes = a.reshape(3, -1)
        assert np.array_equal(planes[0], planes[1]) and np.array_equal(planes[2], planes[1])

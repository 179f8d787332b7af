"""The problems of a batched static step stay apart: a CTA goes from one problem's
tile to another's, and every problem keeps the bits of its own run."""
import numpy as np
import pytest

from paper_2007_05718_gb300 import lbrt
from paper_2007_05718_gb300 import workloads as W

pytestmark = pytest.mark.gpu
P, V = lbrt.LB_RT_PERIODIC, lbrt.LB_RT_VACUUM
F32, F16, BF16 = lbrt.LB_RT_F32, lbrt.LB_RT_F16_DEV, lbrt.LB_RT_BF16_DEV
ICO = [dict(dirset=lbrt.LB_RT_ICOSPHERE, level=l) for l in (0, 1, 2)]
RING = lambda n: dict(dirset=lbrt.LB_RT_RING2D, ndir=n)  # noqa: E731


def _batch(probs, storage, steps, **opts):
    """E, F of every problem (dict: dims, shape, dirs, fluid, state, bc) after `steps`."""
    opts.setdefault("autotune", False)
    b = lbrt.lb_rt_batch_create(max_problems=len(probs), storage=storage, steps_per_tick=steps, **opts)
    try:
        slots = []
        for p in probs:
            nz, ny, nx = p["shape"]
            slots.append(lbrt.lb_rt_batch_admit(
                b, dict(dims=p["dims"], nx=nx, ny=ny, nz=nz, bc=p["bc"], **p["dirs"], **p.get("opts", {})),
                p["fluid"], p["state"], lbrt.LB_RT_STATE_POPULATIONS, steps))
        lbrt.lb_rt_batch_tick(b)
        lbrt.lb_rt_batch_sync(b)
        out = []
        for p, s in zip(probs, slots):
            E, F = np.zeros(p["shape"], np.float32), np.zeros((3,) + p["shape"], np.float32)
            lbrt.lb_rt_batch_moments(b, s, E, F)
            out.append((E, F))
        return out, [lbrt.lb_rt_batch_plan(b, s) for s in slots]
    finally:
        lbrt.lb_rt_batch_destroy(b)


def _alone(p, storage, steps):
    nz, ny, nx = p["shape"]
    h = lbrt.lb_rt_create(p["dims"], nx, ny, nz, storage=storage, bc=p["bc"], **p["dirs"], **p.get("opts", {}))
    try:
        lbrt.lb_rt_set_fluid(h, **p["fluid"])
        lbrt.lb_rt_set_state(h, p["state"])
        lbrt.lb_rt_step(h, steps)
        E, F = np.zeros(p["shape"], np.float32), np.zeros((3,) + p["shape"], np.float32)
        lbrt.lb_rt_moments(h, E, F)
        return E, F
    finally:
        lbrt.lb_rt_destroy(h)


@pytest.mark.parametrize("storage", [F32, F16])
@pytest.mark.parametrize("dims,shape,dirs,ndir", [(3, (2, 70, 40), ICO[0], 12), (2, (1, 600, 20), RING(24), 24)],
                         ids=["3D", "2D"])
def test_batch_of_many_short_tiles(cuda, storage, dims, shape, dirs, ndir):
    """Tiles of one or two batches and a new problem with other fields, steps and
    buffers every few tiles: each CTA turns its tile queue over many times."""
    probs = [dict(dims=dims, shape=shape, dirs=dirs, bc=(P, V, P), fluid=dict(kappa_a=0.5 + k, eta=1.0 + k),
                  state=W.random_populations(ndir, shape, 100 + k)) for k in range(60)]
    got, _ = _batch(probs, storage, 3, use_graph=False)
    for p, (E, F) in zip(probs, got):
        E1, F1 = _alone(p, storage, 3)
        assert np.array_equal(E, E1) and np.array_equal(F, F1)


@pytest.mark.parametrize("storage", [F32, F16, BF16])
@pytest.mark.parametrize("lam", [0.0, 0.3])
def test_non_finite_2d_problem_stays_alone(cuda, storage, lam):
    """A diverged 2D problem of a batch reaches no other one, though its tiles
    and theirs go through the same CTAs (1024 tiles, one or two CTAs an SM)."""
    shape = (1, 2048, 66)
    probs = [dict(dims=2, shape=shape, dirs=RING(120), bc=(P, P, P), fluid=dict(kappa_0=2.0 + k, lam=lam),
                  state=W.random_populations(120, shape, k)) for k in range(4)]
    probs[0]["state"][:] = np.inf
    got, _ = _batch(probs, storage, 2)
    assert not np.isfinite(got[0][0]).any()
    for p, (E, F) in list(zip(probs, got))[1:]:
        E1, F1 = _alone(p, storage, 2)
        assert np.isfinite(E1).all()
        assert np.array_equal(E, E1) and np.array_equal(F, F1)


@pytest.mark.parametrize("storage", [F32, F16, BF16])
def test_non_finite_rows_of_a_2d_grid_reach_their_neighbours_only(cuda, storage):
    """One step moves a value by one row at most, whichever CTA ran which tile."""
    ny, nx = 640, 1024
    h = lbrt.lb_rt_create(2, nx, ny, 1, storage=storage, bc=(P, V, P), **RING(120))
    try:
        lbrt.lb_rt_set_fluid(h, kappa_0=1.0)
        E = []
        for bad in (False, True):
            E0 = W.random_fields((1, ny, nx), 5, 0.5, 1.5)
            if bad:
                E0[0, :ny // 2] = np.inf
            lbrt.lb_rt_set_state(h, E0, lbrt.LB_RT_STATE_ISOTROPIC)
            lbrt.lb_rt_step(h, 1)
            E.append(np.zeros((1, ny, nx), np.float32))
            lbrt.lb_rt_moments(h, E[-1])
    finally:
        lbrt.lb_rt_destroy(h)
    far = ny // 2 + 1
    assert np.isfinite(E[0]).all()
    assert not np.isfinite(E[1][0, :far]).any()
    assert np.array_equal(E[0][0, far:], E[1][0, far:])


def test_every_batched_kernel_gets_its_own_residency(cuda):
    """42 float32 directions: the autotuner times the alternative kernel (one
    plane a batch, 72 registers, three CTAs of nine warps an SM) on its fifth
    tick, and with more CTAs than the plan's own kernel (two of 96 registers)."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shape = (64, 256, 64)  # 512 tiles or more, whatever the z chunk
    b = lbrt.lb_rt_batch_create(max_problems=2, storage=F32, steps_per_tick=1)
    try:
        s = [lbrt.lb_rt_batch_admit(b, dict(dims=3, nx=64, ny=256, nz=64, **ICO[1]), dict(kappa_0=2.0),
                                    W.random_fields(shape, k), lbrt.LB_RT_STATE_ISOTROPIC, 100) for k in range(2)]
        seen = []
        for _ in range(5):
            lbrt.lb_rt_batch_tick(b)
            seen.append((lbrt.lb_rt_batch_plan(b, s[0])[1], lbrt.lb_rt_batch_tuning(b, s[0])[1]))
        lbrt.lb_rt_batch_sync(b)
    finally:
        lbrt.lb_rt_batch_destroy(b)
    assert seen == [(2, 2 * sms)] * 4 + [(1, 3 * sms)]


def test_tuning_and_plan_follow_the_flux_terms(cuda):
    """The flux terms (lambda != 0 somewhere in the group) take one plane a batch
    and have no alternative kernel to time; a tile shape chosen with them is not
    kept once they are gone."""
    b = lbrt.lb_rt_batch_create(max_problems=2, storage=F32, steps_per_tick=1)
    try:
        prob = dict(dims=3, nx=64, ny=16, nz=64, **ICO[1])
        E0 = W.random_fields((64, 16, 64), 1)
        lbrt.lb_rt_batch_admit(b, prob, dict(kappa_0=2.0, lam=0.3), E0, lbrt.LB_RT_STATE_ISOTROPIC, 6)
        s = lbrt.lb_rt_batch_admit(b, prob, dict(kappa_0=2.0), E0, lbrt.LB_RT_STATE_ISOTROPIC, 100)
        planes = []
        for _ in range(11):
            lbrt.lb_rt_batch_tick(b)
            planes.append(lbrt.lb_rt_batch_plan(b, s)[1])
        lbrt.lb_rt_batch_sync(b)
    finally:
        lbrt.lb_rt_batch_destroy(b)
    # six ticks with the flux terms; then four z chunks and the alternative kernel
    assert planes == [1] * 6 + [2] * 4 + [1]


def test_flux_terms_do_not_keep_groups_from_pairing(cuda):
    b = lbrt.lb_rt_batch_create(max_problems=2, storage=F32, steps_per_tick=1, pair_groups=1)
    try:
        E0 = W.random_fields((16, 16, 64), 1)
        s = [lbrt.lb_rt_batch_admit(b, dict(dims=3, nx=64, ny=16, nz=16, **ICO[l]), dict(kappa_0=2.0, lam=0.3),
                                    E0, lbrt.LB_RT_STATE_ISOTROPIC, 100) for l in (1, 2)]
        paired = []
        for _ in range(6):
            lbrt.lb_rt_batch_tick(b)
            paired.append([lbrt.lb_rt_batch_plan(b, k)[2] for k in s])
        lbrt.lb_rt_batch_sync(b)
    finally:
        lbrt.lb_rt_batch_destroy(b)
    assert paired == [[0, 0]] * 4 + [[1, 1]] * 2


@pytest.mark.parametrize("storage", [F32, F16, BF16])
@pytest.mark.parametrize("lams", [(0.3, 0.0), (0.0, 0.3), (0.3, 0.3)], ids=str)
def test_paired_launch_with_flux_terms(cuda, storage, lams):
    """A lambda in either group puts both on the flux terms of the paired kernel,
    the 42-direction group on its one-plane boxes."""
    probs = []
    for k, (shape, level, ndir) in enumerate([((9, 5, 63), 1, 42), ((12, 3, 65), 2, 162), ((17, 4, 64), 1, 42),
                                              ((3, 7, 130), 2, 162)]):
        probs.append(dict(dims=3, shape=shape, dirs=ICO[level], bc=(P, V, P), state=W.random_populations(ndir, shape, k),
                          fluid=dict(kappa_a=0.5, kappa_0=3.0, eta=W.random_fields(shape, 9 + k),
                                     lam=lams[0] if level == 1 and k == 0 else lams[1] if level == 2 and k == 1 else 0.0)))
    got, plans = _batch(probs, storage, 5, pair_groups=1)
    assert plans == [(5, 1, 1), (11, 1, 1)] * 2
    for p, (E, F) in zip(probs, got):
        E1, F1 = _alone(p, storage, 5)
        assert np.isfinite(E1).all() and np.array_equal(E, E1) and np.array_equal(F, F1)

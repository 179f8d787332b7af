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

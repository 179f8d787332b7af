"""Performance cases of the radiative Lattice-Boltzmann library.

A case is one situation of real use: a handle (or a batch of problems) that a
program keeps, and a pass that advances it by some steps through the public
entry points of paper_2007_05718_gb300.lbrt and reads back what such a program
reads: the moments E and F (with the coupling outputs, the populations or the
energy budget where the program uses them).  Inputs are made from a seed on
the GPU; every output has a float64 counterpart from `exact`, which is plain
torch and shares no code with the library.

Kinds of case:
  diffusion  optically thick scattering, periodic faces, uniform kappa_0
  sphere     an emitting and absorbing ball in vacuum, per-site kappa_a and eta
  shear      moving fluid (mixed frame), per-site velocity and opacities
  coupled    a fluid code that hands new per-site opacities over every step and
             takes E, F and the four-force back
  beam       2D beam injection: frozen cells, vacuum in x, no interaction
  general    ragged grid, mixed faces, lambda != 0, a product quadrature, the
             paper's Lambda iteration or the explicit step, the energy budget
  serving    many problems of uneven size in one batch
  sweep      2D diffusion-coefficient sweep, many points in one batch
"""
import math

import numpy as np
import torch

from paper_2007_05718_gb300 import lbrt

P, V = lbrt.LB_RT_PERIODIC, lbrt.LB_RT_VACUUM
STORAGE = {"f32": lbrt.LB_RT_F32, "f16": lbrt.LB_RT_F16_DEV, "bf16": lbrt.LB_RT_BF16_DEV}
COLLISION = {"implicit": lbrt.LB_RT_IMPLICIT_EXACT, "explicit": lbrt.LB_RT_EXPLICIT,
             "lambda": lbrt.LB_RT_LAMBDA_K}
DEV = "cuda"


def listed():
    return [
        # the optically thick diffusion problem at full size, each storage a user picks for it
        dict(name="diffusion 256 f32", kind="diffusion", nx=256, ny=256, nz=256, level=2,
             storage="f32", steps=8),
        dict(name="diffusion 256 f16", kind="diffusion", nx=256, ny=256, nz=256, level=2,
             storage="f16", steps=8),
        # bfloat16 where it is validated (scattering), a middle-sized box
        dict(name="diffusion 96 bf16", kind="diffusion", nx=96, ny=96, nz=96, level=2,
             storage="bf16", steps=20),
        # the radiating sphere: 42 directions, vacuum faces, per-site fields
        dict(name="sphere 128 f32", kind="sphere", nx=128, ny=128, nz=128, level=1,
             storage="f32", steps=40),
        dict(name="sphere 128 f16", kind="sphere", nx=128, ny=128, nz=128, level=1,
             storage="f16", steps=40),
        # moving background fluid, both storages
        dict(name="shear 192 f32", kind="shear", nx=192, ny=192, nz=192, level=2,
             storage="f32", steps=6),
        dict(name="shear 128 f16", kind="shear", nx=128, ny=128, nz=128, level=2,
             storage="f16", steps=10),
        # coupled to a fluid code on the same GPU: new fields and outputs every step
        dict(name="coupled 64 f32", kind="coupled", nx=64, ny=64, nz=64, level=1,
             storage="f32", steps=10),
        # 2D beam: the smallest problems, hundreds of tiny steps
        dict(name="beam 64 f32", kind="beam", nx=64, ny=64, nz=1, ndir=16, storage="f32", steps=100),
        # the general path: ragged, mixed faces, flux term, product quadrature
        dict(name="general 93x61x47 f32", kind="general", nx=93, ny=61, nz=47, gl_theta=6, gl_phi=12,
             storage="f32", steps=20, collision="lambda", iters=5, bc="pvv"),
        # continuous batching: spheres of uneven size and direction count, FP16
        dict(name="serving mix f16", kind="serving", problems=10, largest=128, storage="f16", steps=40),
        # the 2D sweep of kappa_0, cfl and lambda in one batch
        dict(name="sweep 512 f32", kind="sweep", problems=8, nx=512, ny=512, ndir=120,
             storage="f32", steps=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["diffusion", "diffusion", "sphere", "sphere", "shear", "coupled", "beam",
                       "general", "serving", "sweep"])
    if kind == "beam":
        return dict(kind=kind, nx=_log_int(rng, 32, 400), ny=_log_int(rng, 24, 300), nz=1,
                    ndir=2 * rng.randint(4, 60), storage="f32", steps=rng.randint(20, 100))
    if kind == "serving":
        return dict(kind=kind, problems=rng.randint(2, 16), largest=rng.choice([64, 96, 128]),
                    storage=rng.choice(["f16", "f16", "f32"]), steps=rng.randint(10, 50))
    if kind == "sweep":
        return dict(kind=kind, problems=rng.randint(2, 10), nx=_log_int(rng, 96, 512),
                    ny=_log_int(rng, 96, 512), ndir=2 * rng.randint(8, 60), storage="f32",
                    steps=rng.randint(5, 25))
    if kind == "general":
        theta, phi = rng.choice([(4, 8), (6, 12), (8, 16)])
        return dict(kind=kind, nx=rng.randint(17, 140), ny=rng.randint(9, 90), nz=rng.randint(5, 70),
                    gl_theta=theta, gl_phi=phi, storage="f32", steps=rng.randint(4, 24),
                    collision=rng.choice(["implicit", "explicit", "lambda"]), iters=rng.randint(1, 8),
                    bc="".join(rng.choice("pv") for _ in range(3)))
    top = {"diffusion": 224, "sphere": 224, "shear": 176, "coupled": 160}[kind]
    storage = {"diffusion": ["f32", "f16", "bf16"], "sphere": ["f32", "f16"], "shear": ["f32", "f16"],
               "coupled": ["f32"]}[kind]
    nx, ny, nz = (_log_int(rng, 24, top) for _ in range(3))
    if rng.random() < 0.5:  # half of them have whole rows, as most users choose them
        nx = max(32, nx // 32 * 32)
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, level=rng.choice([1, 2]), storage=rng.choice(storage),
                steps=rng.randint(3, 10))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _rng(seed):
    return np.random.default_rng([int(seed), 20200711])


def _grid(nx, ny, nz, dx):
    ax = lambda n: (torch.arange(n, device=DEV, dtype=torch.float32) + 0.5) * dx  # noqa: E731
    return ax(nx)[None, None, :], ax(ny)[None, :, None], ax(nz)[:, None, None]


def _smooth(shape, g, modes=6):
    """Sum of seeded Fourier modes of the box, in [-1, 1]."""
    nz, ny, nx = shape
    x, y, z = (torch.arange(n, device=DEV, dtype=torch.float32) * (2 * math.pi / n) for n in (nx, ny, nz))
    out = torch.zeros(shape, device=DEV)
    for _ in range(modes):
        kx, ky, kz = (int(v) for v in g.integers(1, 4, size=3))
        ph = float(g.uniform(0, 2 * math.pi))
        out += torch.sin(kx * x[None, None, :] + ky * y[None, :, None] + kz * z[:, None, None] + ph)
    return out / modes


def _ball(nx, ny, nz, centre, R):
    """Distance from `centre` over R, box lengths in units of nx cells."""
    dx = 1.0 / nx
    x, y, z = _grid(nx, ny, nz, dx)
    r2 = (x - centre[0]) ** 2 + (y - centre[1] * ny * dx) ** 2 + (z - centre[2] * nz * dx) ** 2
    return torch.sqrt(r2) / R


def _gaussian(nx, ny, nz, g, sigma=8.0):
    c = g.uniform(0.3, 0.7, size=3)
    x, y, z = _grid(nx, ny, nz, 1.0)
    r2 = (x - c[0] * nx) ** 2 + (y - c[1] * ny) ** 2 + (z - c[2] * nz) ** 2
    return (float(g.uniform(0.5, 2.0)) * torch.exp(-r2 / (2 * sigma * sigma))).contiguous()


def _sphere_fields(nx, ny, nz, g):
    """An emitting ball (kappa_a = eta) in vacuum and its isotropic E0; every
    other one with a black absorber in front (the shadow problem)."""
    c = g.uniform(0.4, 0.6, size=3)
    R = 0.25 * min(nx, ny, nz) / nx
    kappa = float(10.0 ** g.uniform(0.0, 2.5))
    r = _ball(nx, ny, nz, c, R)
    ka = torch.where(r < 1.0, kappa, 0.0)
    eta = ka.clone()
    if g.random() < 0.5:
        c2 = (c[0] + 0.35 * (1 if c[0] < 0.5 else -1), c[1], c[2])
        ra = _ball(nx, ny, nz, c2, 0.5 * R)
        ka = torch.where(ra < 1.0, 1e4, ka)
        eta = torch.where(ra < 1.0, 0.0, eta)
    E0 = torch.clamp(1.0 / (r * r), max=1.0)
    return ka.contiguous(), eta.contiguous(), E0.contiguous()


def _problem(case, seed):
    """Everything the library and the float64 counterpart need, as a dict:
    dims, (nz, ny, nx), dirs (kind), cfl, dx, bc, collision, coef, state."""
    g = _rng(seed)
    kind = case["kind"]
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape = (nz, ny, nx)
    p = dict(dims=2 if nz == 1 and kind == "beam" else 3, shape=shape, cfl=0.5, dx=1.0 / nx, bc=(P, P, P),
             collision="implicit", iters=1, moving=False, budget=False, frozen=None,
             storage=case["storage"], dirs=("ico", case.get("level", 1)))
    if kind == "diffusion":
        p["coef"] = dict(kappa_0=float(g.uniform(3.0, 4.5)) * nx)
        p["E0"] = _gaussian(nx, ny, nz, g)
    elif kind == "sphere":
        ka, eta, E0 = _sphere_fields(nx, ny, nz, g)
        p.update(coef=dict(kappa_a=ka, eta=eta), E0=E0, bc=(V, V, V))
    elif kind == "shear":
        y = (torch.arange(ny, device=DEV, dtype=torch.float32) + 0.5) / ny
        vx = 0.5 * (torch.tanh((y - 0.25) / 0.02) - torch.tanh((y - 0.75) / 0.02) - 1.0)
        v = torch.stack([vx[None, :, None].expand(shape) + 0.05 * _smooth(shape, g),
                         0.1 * _smooth(shape, g), 0.1 * _smooth(shape, g)])
        s = torch.sqrt((v * v).sum(0))
        v *= torch.where(s > 0.6, 0.6 / s, 1.0)[None]
        rho = 0.5 * (1.0 + _smooth(shape, g))
        kta = 0.1 * 1000.0 ** rho
        p.update(moving=True, E0=1.0 + 0.3 * _smooth(shape, g),
                 coef=dict(v=v.contiguous(), kt_a=kta, kt_0=100.0 * rho, eta_t=kta.clone()))
    elif kind == "coupled":
        p["E0"] = 1.0 + 0.3 * _smooth(shape, g)
        ka, k0 = 5.0 + 4.0 * _smooth(shape, g), 20.0 + 15.0 * _smooth(shape, g)
        # the fluid code's fields of every step (it would compute them from S)
        p["series"] = [(ka * (1.0 + 0.02 * k), k0 * (1.0 - 0.02 * k), ka * (1.0 + 0.01 * k))
                       for k in range(case["steps"])]
        p["coef"] = dict()
    elif kind == "beam":
        n = case["ndir"]
        p.update(dirs=("ring", n), coef=dict(), cfl=0.2, bc=(V, P, P))
        p["I0"] = torch.zeros((n,) + shape, device=DEV)
        ys = np.arange(ny // 4, ny - ny // 4)
        vals = np.zeros((len(ys), n), dtype=np.float32)
        vals[:, 0] = g.uniform(0.5, 1.5, size=len(ys))
        vals[:, 1] = g.uniform(0.1, 0.5, size=len(ys))
        p["frozen"] = ((ys * nx).astype(np.int64), vals)
    elif kind == "general":
        ka = 8.0 + 6.0 * _smooth(shape, g)
        p.update(dirs=("gl", case["gl_theta"], case["gl_phi"]), collision=case["collision"],
                 iters=case["iters"], bc=tuple(P if c == "p" else V for c in case["bc"]), budget=True,
                 coef=dict(kappa_a=ka, kappa_0=20.0 + 15.0 * _smooth(shape, g),
                           lam=0.5 * _smooth(shape, g), eta=ka * (1.0 + 0.5 * _smooth(shape, g))))
        N = case["gl_theta"] * case["gl_phi"]
        t = torch.Generator(device=DEV).manual_seed(int(g.integers(1 << 30)))
        p["I0"] = torch.rand((N,) + shape, generator=t, device=DEV) / N
    return p


def _serving_sizes(case):
    """The sizes of the request stream's problems, largest first, taken in turn."""
    sizes = [n for n in (128, 96, 64, 48, 32) if n <= case["largest"]]
    return [sizes[k % len(sizes)] for k in range(case["problems"])]


def _batch_problems(case, seed):
    g = _rng(seed)
    out = []
    for k in range(case["problems"]):
        if case["kind"] == "serving":
            n = _serving_sizes(case)[k]
            ka, eta, E0 = _sphere_fields(n, n, n, g)
            out.append(dict(dims=3, shape=(n, n, n), cfl=0.5, dx=1.0 / n, bc=(V, V, V),
                            dirs=("ico", 1 + k % 2), coef=dict(kappa_a=ka, eta=eta), E0=E0))
        else:
            nx, ny = case["nx"], case["ny"]
            out.append(dict(dims=2, shape=(1, ny, nx), cfl=(0.1, 0.25, 0.5, 1.0)[k % 4], dx=1.0, bc=(P, P, P),
                            dirs=("ring", case["ndir"]), E0=_gaussian(nx, ny, 1, g, 10.0),
                            coef=dict(kappa_0=float(g.uniform(0.5, 10.0)), lam=(0.0, 0.25, 0.5, 0.75)[k // 2 % 4])))
        out[-1].update(collision="implicit", iters=1, moving=False, frozen=None)
    return out


# ---------------------------------------------------------------------------
# the library
# ---------------------------------------------------------------------------

def _dir_args(p):
    d = p["dirs"]
    if d[0] == "ico":
        return dict(dirset=lbrt.LB_RT_ICOSPHERE, level=d[1])
    if d[0] == "ring":
        return dict(dirset=lbrt.LB_RT_RING2D, ndir=d[1])
    return dict(dirset=lbrt.LB_RT_GAUSS_LEGENDRE, gl=(d[1], d[2]))


class _State:
    """A handle (or a batch) with the tensors that its program keeps."""

    def __init__(self, free):
        self._free = free

    def __del__(self):
        self._free()


def prepare(case, seed):
    if case["kind"] in ("serving", "sweep"):
        return _prepare_batch(case, seed)
    p = _problem(case, seed)
    nz, ny, nx = p["shape"]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    h = lbrt.lb_rt_create(p["dims"], nx, ny, nz, cfl=p["cfl"], dx=p["dx"], bc=p["bc"],
                          storage=STORAGE[p["storage"]], collision=COLLISION[p["collision"]],
                          lambda_iters=p["iters"], moving=p["moving"], budget=p["budget"],
                          stream=stream.cuda_stream, **_dir_args(p))
    st = _State(lambda: lbrt.lb_rt_destroy(h))
    st.h, st.stream, st.kind, st.steps = h, stream, case["kind"], case["steps"]
    lbrt.lb_rt_set_fluid(h, **p["coef"])
    if "I0" in p:
        lbrt.lb_rt_set_state(h, p["I0"], lbrt.LB_RT_STATE_POPULATIONS)
    else:
        lbrt.lb_rt_set_state(h, p["E0"], lbrt.LB_RT_STATE_ISOTROPIC)
    if p["frozen"] is not None:
        lbrt.lb_rt_set_frozen(h, *p["frozen"])
    st.E = torch.zeros(p["shape"], device=DEV)
    st.F = torch.zeros((3,) + p["shape"], device=DEV)
    if case["kind"] == "coupled":
        st.series = p["series"]
        st.J = torch.zeros_like(st.E)
        st.H = torch.zeros_like(st.F)
        st.S = torch.zeros((4,) + p["shape"], device=DEV)
    if case["kind"] in ("beam", "general"):
        st.I = torch.zeros_like(p["I0"])
    lbrt.lb_rt_sync(h)
    torch.cuda.synchronize()
    return st


def _prepare_batch(case, seed):
    probs = _batch_problems(case, seed)
    torch.cuda.synchronize()
    b = lbrt.lb_rt_batch_create(max_problems=len(probs), storage=STORAGE[case["storage"]],
                                steps_per_tick=case["steps"], mem_budget=60 << 30,
                                pair_groups=2 if case["kind"] == "serving" else 0)
    st = _State(lambda: lbrt.lb_rt_batch_destroy(b))
    st.b, st.kind, st.keep, st.out = b, case["kind"], probs, []
    for p in probs:
        nz, ny, nx = p["shape"]
        slot = lbrt.lb_rt_batch_admit(b, dict(dims=p["dims"], nx=nx, ny=ny, nz=nz, cfl=p["cfl"], dx=p["dx"],
                                              bc=p["bc"], **_dir_args(p)),
                                      p["coef"], p["E0"], lbrt.LB_RT_STATE_ISOTROPIC, 1 << 40)
        st.out.append((slot, torch.zeros(p["shape"], device=DEV), torch.zeros((3,) + p["shape"], device=DEV)))
    torch.cuda.synchronize()
    return st


def run(st):
    if st.kind in ("serving", "sweep"):
        # one tick of every resident problem, then the fields of each
        lbrt.lb_rt_batch_tick(st.b)
        for slot, E, F in st.out:
            lbrt.lb_rt_batch_moments(st.b, slot, E, F)
        return [(E, F) for _, E, F in st.out]
    if st.kind == "coupled":
        for ka, k0, eta in st.series:
            lbrt.lb_rt_set_fluid(st.h, kappa_a=ka, kappa_0=k0, lam=0.3, eta=eta)
            lbrt.lb_rt_step_moments(st.h, 1, st.E, st.F)
            lbrt.lb_rt_coupling(st.h, st.J, st.H, st.S)
        return dict(E=st.E, F=st.F, J=st.J, H=st.H, S=st.S)
    lbrt.lb_rt_step(st.h, st.steps)
    if st.kind == "general":
        b = lbrt.lb_rt_moments(st.h, st.E, st.F, budget=True)
        lbrt.lb_rt_get_populations(st.h, st.I)
        return dict(E=st.E, F=st.F, I=st.I, total=b["total"], source=b["source"], steps=b["steps"])
    lbrt.lb_rt_moments(st.h, st.E, st.F)
    if st.kind == "beam":
        lbrt.lb_rt_get_populations(st.h, st.I)
        return dict(E=st.E, F=st.F, I=st.I)
    return dict(E=st.E, F=st.F)


# ---------------------------------------------------------------------------
# work of a pass
# ---------------------------------------------------------------------------

def _ndir(case):
    if "gl_theta" in case:
        return case["gl_theta"] * case["gl_phi"]
    return case["ndir"] if "ndir" in case else 10 * 4 ** case["level"] + 2


def work(case):
    """Every step reads and writes the populations once (4 bytes each, or 2
    and a float32 E per site) and reads its per-site fields; the outputs are
    written once.  About 23 flops a site and direction for the interpolation,
    the moments and the collision (12 more with a flux term or a moving
    fluid)."""
    kind = case["kind"]
    pop = 8.0 if case["storage"] == "f32" else 4.0
    esite = 0.0 if case["storage"] == "f32" else 8.0
    if kind == "serving":
        sites = [n ** 3 for n in _serving_sizes(case)]
        ndir = [(42, 162)[k % 2] for k in range(len(sites))]
        return dict(bytes=sum(s * (case["steps"] * (N * pop + esite + 8) + 16) for s, N in zip(sites, ndir)),
                    flops=sum(s * case["steps"] * N * 23 for s, N in zip(sites, ndir)))
    N = _ndir(case)
    if kind == "sweep":
        sites = case["problems"] * case["nx"] * case["ny"]
        return dict(bytes=sites * (case["steps"] * N * pop + 16), flops=sites * case["steps"] * N * 35)
    sites = case["nx"] * case["ny"] * case["nz"]
    fields = {"sphere": 8, "shear": 24, "coupled": 12, "general": 16}.get(kind, 0)
    out = {"coupled": 48 * case["steps"], "beam": 16 + 4 * N, "general": 16 + 4 * N}.get(kind, 16)
    flops = 35 if kind in ("shear", "coupled", "general") else 23
    return dict(bytes=sites * (case["steps"] * (N * pop + esite + fields) + out),
                flops=sites * case["steps"] * N * flops)


# ---------------------------------------------------------------------------
# the same in 64 bits: plain torch
# ---------------------------------------------------------------------------

def _icosphere(level):
    phi = (1.0 + math.sqrt(5.0)) / 2.0
    v = []
    for a in (-1.0, 1.0):
        for b in (-phi, phi):
            v += [(0.0, a, b), (a, b, 0.0), (b, 0.0, a)]
    v = np.array(v)
    d = np.linalg.norm(v[:, None] - v[None], axis=-1)
    faces = [(a, b, c) for a in range(12) for b in range(a + 1, 12) for c in range(b + 1, 12)
             if max(abs(d[a, b] - 2), abs(d[b, c] - 2), abs(d[a, c] - 2)) < 1e-6]
    pts = [tuple(x / np.linalg.norm(x)) for x in v]
    for _ in range(level):
        mids, finer = {}, []

        def mid(a, b):
            k = (min(a, b), max(a, b))
            if k not in mids:
                m = np.array(pts[a]) + np.array(pts[b])
                mids[k] = len(pts)
                pts.append(tuple(m / np.linalg.norm(m)))
            return mids[k]

        for a, b, c in faces:
            ab, bc, ca = mid(a, b), mid(b, c), mid(c, a)
            finer += [(a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca)]
        faces = finer
    n = np.array(pts)
    return n, np.full(len(n), 1.0 / len(n))


def _directions(d):
    """Unit vectors and weights, sorted by (n_z, n_y, n_x) in 3D as the
    library numbers its directions."""
    if d[0] == "ring":
        a = 2 * math.pi * np.arange(d[1]) / d[1]
        n, w = np.stack([np.cos(a), np.sin(a), 0 * a], 1), np.full(d[1], 1.0 / d[1])
        n[np.abs(n) < 1e-15] = 0.0
        return n, w
    if d[0] == "ico":
        n, w = _icosphere(d[1])
    else:
        mu, wm = np.polynomial.legendre.leggauss(d[1])
        a = 2 * math.pi * (np.arange(d[2]) + 0.5) / d[2]
        s = np.sqrt(1 - mu * mu)
        n = np.stack([np.outer(s, np.cos(a)), np.outer(s, np.sin(a)), np.outer(mu, np.ones(d[2]))], -1).reshape(-1, 3)
        w = np.repeat(wm / 2.0 / d[2], d[2])
    n[np.abs(n) < 1e-15] = 0.0
    k = np.rint(n * 1e9).astype(np.int64)
    order = np.lexsort((k[:, 0], k[:, 1], k[:, 2]))
    return n[order], w[order]


def _pull(f, s, axis, bc):
    g = torch.roll(f, s, dims=axis)
    if bc == V:
        g.select(axis, 0 if s > 0 else -1).zero_()
    return g


def _step64(I, n, w, p, c):
    """One step in place; returns sum(E*) and sum(E) after the collision."""
    dt, d = p["cfl"] * p["dx"], p["dims"]
    for i in range(len(w)):
        f = I[i]
        for a in range(d):
            if n[i, a] != 0.0:
                s = 1 if n[i, a] > 0 else -1
                f = torch.lerp(f, _pull(f, s, 2 - a, p["bc"][a]), p["cfl"] * abs(n[i, a]))
        I[i] = f
    if p["moving"]:
        v, kta, kt0, et = c["v"], c["kt_a"], c["kt_0"], c["eta_t"]
        W = 1.0 / torch.sqrt(1.0 - (v * v).sum(0))
        X, Y = torch.zeros_like(W), torch.zeros_like(W)
        terms = lambda i: _moving_terms(W, v, n[i], w[i], dt, kta, kt0)  # noqa: E731
        for i in range(len(w)):
            b, A, D = terms(i)
            X += b * b * A * (I[i] + dt * D * et)
            Y += b * b * A * D
        J = W * W * X / (1.0 - dt * kt0 * W * W * Y)
        for i in range(len(w)):
            b, A, D = terms(i)
            I[i] = A * (I[i] + dt * D * (et + kt0 * J))
        return None
    ka, k0, lam, eta = c["kappa_a"], c["kappa_0"], c["lam"], c["eta"]
    E, F = _moments64(I, n, d)
    src = E.sum()
    A = 1.0 / (1.0 + dt * (k0 + ka))
    if p["collision"] == "implicit":
        E = (E + dt * eta) / (1.0 + dt * ka)
        F = F / (1.0 + dt * (k0 + ka) - dt * k0 * lam / d)
    elif p["collision"] == "lambda":
        E0, F0 = E, F
        for _ in range(p["iters"] - 1):
            E = A * (E0 + dt * eta + dt * k0 * E)
            F = A * (F0 + dt * k0 * lam * F / d)
    for i in range(len(w)):
        nF = sum(n[i, a] * F[a] for a in range(d))
        if p["collision"] == "explicit":
            I[i] = I[i] - k0 * dt * (I[i] - w[i] * (E + lam * nF)) + dt * (w[i] * eta - ka * I[i])
        else:
            I[i] = A * (I[i] + dt * w[i] * eta + dt * k0 * w[i] * (E + lam * nF))
    return I.sum() - src


def _moving_terms(W, v, n, w, dt, kta, kt0):
    b = 1.0 - (n[0] * v[0] + n[1] * v[1] + n[2] * v[2])
    return b, 1.0 / (1.0 + dt * W * b * (kta + kt0)), w / (W * b) ** 3


def _moments64(I, n, d=3):
    E = I.sum(0)
    F = torch.zeros((3,) + tuple(E.shape), dtype=E.dtype, device=E.device)
    for i in range(len(n)):
        for a in range(d):
            F[a] += n[i, a] * I[i]
    return E, F


def _start64(p):
    n, w = _directions(p["dirs"])
    if "I0" in p:
        return n, w, p["I0"].double()
    I = torch.empty((len(w),) + tuple(p["shape"]), dtype=torch.float64, device=DEV)
    for i in range(len(w)):
        I[i] = w[i] * p["E0"].double()
    return n, w, I


def _coef64(p, coef):
    zero = dict(kt_a=0.0, kt_0=0.0, eta_t=0.0) if p["moving"] else dict(kappa_a=0.0, kappa_0=0.0, lam=0.0, eta=0.0)
    f32 = lambda x: x.double() if torch.is_tensor(x) else float(np.float32(x))  # noqa: E731
    return {k: f32(x) for k, x in {**zero, **coef}.items()}


def _solve64(p, steps):
    """(E, F, I, sum of the collision's sources) after `steps` steps."""
    n, w, I = _start64(p)
    c, src = _coef64(p, p["coef"]), 0.0
    for _ in range(steps):
        s = _step64(I, n, w, p, c)
        src += 0.0 if s is None else float(s)
        if p["frozen"] is not None:
            cells, vals = p["frozen"]
            I.view(len(w), -1)[:, torch.from_numpy(cells).to(DEV)] = torch.from_numpy(vals).to(DEV).double().T
    E, F = _moments64(I, n, p["dims"])
    return E, F, I, src


def exact(case, seed):
    if case["kind"] in ("serving", "sweep"):
        return [_solve64(p, case["steps"])[:2] for p in _batch_problems(case, seed)]
    p = _problem(case, seed)
    if case["kind"] == "coupled":
        n, w, I = _start64(p)
        for ka, k0, eta in p["series"]:
            c = _coef64(p, dict(kappa_a=ka, kappa_0=k0, lam=0.3, eta=eta))
            _step64(I, n, w, p, c)
        E, F = _moments64(I, n)
        kt = c["kappa_a"] + c["kappa_0"]
        S = torch.cat([(c["kappa_a"] * E - c["eta"])[None], kt[None] * F])
        return dict(E=E, F=F, J=E, H=F, S=S)
    E, F, I, src = _solve64(p, case["steps"])
    if case["kind"] == "general":
        return dict(E=E, F=F, I=I, total=float(I.sum()), source=src, steps=None)
    if case["kind"] == "beam":
        return dict(E=E, F=F, I=I)
    return dict(E=E, F=F)

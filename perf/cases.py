"""Performance cases of the framework: what a user's program runs, through the
public Python entry points (Lattice, InPlaceLattice, Batch, Surrogate and the
lbm_* functions beside them).

A case is one dict of plain values; `kind` selects the path:
  lattice  one two-buffer lattice: `steps` time steps, then what the program
           reads back: the moment fields (`read` = "moments"), these and the
           populations ("state"), or the raw checkpoint ("checkpoint", the
           16-bit formats' own values)
  inplace  one lattice stepped in place on a single population array
  batch    many independent lattices advanced together
  predict  inference of the spreading-factor network
  train    Adam steps of that network on minibatches already on the GPU
`scene` is the physical set-up of a lattice: a droplet in a uniform stream, a
layered channel driven by a force, a Rayleigh-Taylor column, a drop falling
onto a wetted floor.  Flows are set moving from the start, as in a run under
way, so that velocities are well above the rounding of their sums.
"""
import math

import numpy as np
import torch

from paper_1904_03618_gb300 import lbm
from paper_1904_03618_gb300 import params as P
from paper_1904_03618_gb300 import rt as RT
from paper_1904_03618_gb300 import surrogate as S
from paper_1904_03618_gb300 import workloads as W


def listed():
    return [
        # the layered channel of the viscosity-ratio study: the smallest
        # lattice in use, bounce-back walls in y, a body force; one output
        # interval of 100 steps, launches and latency
        dict(name="channel_4x128x4", kind="lattice", scene="channel", nx=4, ny=128, nz=4,
             storage="f32", collision="mrt", steps=100, read="state"),
        # the validation droplet: a lattice of one CTA wave, launch-bound
        dict(name="droplet_32", kind="lattice", scene="droplet", nx=32, ny=32, nz=32,
             storage="f32", collision="mrt", steps=50, read="state"),
        # the 128^3 moving droplet of the benchmark, single and half precision
        dict(name="droplet_128", kind="lattice", scene="droplet", nx=128, ny=128, nz=128,
             storage="f32", collision="mrt", steps=30, read="moments"),
        dict(name="droplet_128_f16", kind="lattice", scene="droplet", nx=128, ny=128, nz=128,
             storage="f16", collision="mrt", steps=30, read="checkpoint"),
        # the benchmark's headline lattice: the largest two-buffer run
        dict(name="rt_256x256x1024", kind="lattice", scene="rt", nx=256, ny=256, nz=1024,
             storage="f32", collision="mrt", steps=8, read="moments"),
        # the same case one size down in BF16 deviation storage
        dict(name="rt_192x192x768_bf16", kind="lattice", scene="rt", nx=192, ny=192, nz=768,
             storage="bf16", collision="mrt", steps=8, read="checkpoint"),
        # a drop impact in a closed box of odd extents: walls on every axis,
        # the contact-angle rule, no 16-byte rows
        dict(name="impact_101x99x67", kind="lattice", scene="impact", nx=101, ny=99, nz=67,
             storage="f32", collision="mrt", steps=20, read="state"),
        # the in-place step, used where two buffers would not fit
        dict(name="inplace_rt_192x192x768", kind="inplace", scene="rt", nx=192, ny=192, nz=768,
             storage="f32", collision="mrt", steps=8),
        # training data of the surrogate: equal boxes with a floor, wetting
        dict(name="batch_impacts_128", kind="batch", scene="impacts", ncases=128, nx=64, ny=64,
             nz=32, storage="f32", steps=12),
        # the droplet parameter sweep: boxes of 32 to 96 cells, half precision
        dict(name="batch_sweep_48_f16", kind="batch", scene="sweep", ncases=48, extra=0,
             storage="f16", steps=12),
        # screening a sweep with the trained network
        dict(name="predict_65536", kind="predict", rows=65536, width=256, depth=4, n_out=16),
        # training it: minibatches of 256
        dict(name="train_256", kind="train", rows=256, width=256, depth=4, n_out=16, steps=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "lattice", "inplace", "batch", "predict",
                       "train"])
    if kind == "predict":
        return dict(kind=kind, rows=_log(rng, 1, 65536), width=rng.choice([64, 96, 128, 200, 256]),
                    depth=rng.randint(1, 4), n_out=rng.choice([8, 16, 24]))
    if kind == "train":
        return dict(kind=kind, rows=_log(rng, 32, 4096), width=rng.choice([64, 128, 256]),
                    depth=rng.randint(1, 4), n_out=rng.choice([8, 16, 24]), steps=4)
    storage = rng.choice(["f32", "f32", "f16", "bf16"])
    if kind == "batch":
        if rng.random() < 0.5:
            return dict(kind=kind, scene="impacts", ncases=rng.randint(8, 64),
                        nx=rng.choice([40, 48, 64, 65, 96]), ny=rng.choice([40, 51, 64, 72]),
                        nz=rng.choice([24, 32, 37]), storage=storage, steps=rng.randint(4, 12))
        return dict(kind=kind, scene="sweep", ncases=rng.randint(8, 48),
                    extra=rng.choice([0, 0, 0, 3, 8]), storage=storage, steps=rng.randint(4, 12))
    scene = rng.choice(["droplet", "channel", "rt", "impact"])
    if kind == "inplace":
        scene = rng.choice(["droplet", "rt", "impact"])
    if scene == "channel":
        nx, ny, nz = rng.choice([1, 4, 16]), rng.randint(64, 160), rng.choice([1, 4, 16, 33])
    elif scene == "rt":
        nx = _log(rng, 24, 160)
        ny, nz = nx, 4 * nx
    else:
        nx, ny, nz = (_log(rng, 24, 224) for _ in range(3))
    steps = 2 * max(2, min(10, 100_000_000 // (nx * ny * nz)))
    c = dict(kind=kind, scene=scene, nx=nx, ny=ny, nz=nz, storage=storage,
             collision="bgk" if rng.random() < 0.1 else "mrt", steps=steps)
    if kind == "lattice":
        c["read"] = "checkpoint" if storage != "f32" else rng.choice(["moments", "state"])
    return c


# ---------------------------------------------------------------------------
# set-ups
# ---------------------------------------------------------------------------
def _dev():
    return torch.device("cuda")


def _axes(nx, ny, nz):
    f = dict(dtype=torch.float64, device=_dev())
    return (torch.arange(nx, **f)[None, None, :], torch.arange(ny, **f)[None, :, None],
            torch.arange(nz, **f)[:, None, None])


def _waves(nx, ny, nz, rng, amp):
    """A smooth periodic velocity disturbance, (3, nz, ny, nx) float32."""
    x, y, z = _axes(nx, ny, nz)
    u = torch.zeros((3, nz, ny, nx), dtype=torch.float32, device=_dev())
    for a in range(3):
        p = rng.uniform(0, 2 * math.pi, 3)
        u[a] = (amp * torch.sin(2 * math.pi * x / nx + p[0]) * torch.cos(2 * math.pi * y / ny + p[1])
                * torch.cos(2 * math.pi * z / nz + p[2])).float()
    return u


def _two_colours(inside, rho_R, rho_B):
    return (torch.where(inside, rho_R, 0.0).float(), torch.where(inside, 0.0, rho_B).float())


def _droplet(nx, ny, nz, rng, pd, speed):
    x, y, z = _axes(nx, ny, nz)
    c = [(n - 1) / 2.0 + rng.uniform(-2, 2) for n in (nx, ny, nz)]
    R = min(nx, ny, nz) * rng.uniform(0.23, 0.27)
    inside = (x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2 <= R * R
    rR, rB = _two_colours(inside, pd["rho_in_R"], pd["rho_in_B"])
    u = _waves(nx, ny, nz, rng, 0.003)
    u[0] += speed
    return rR, rB, u


def _impact_scene(nx, ny, nz, sample):
    """Drop impact of the surrogate's set-up in a box of this size."""
    setup = S.ImpactSetup(radius=max(5, min(nx, ny, 2 * nz) // 8), box=(nx, ny, nz))
    return setup, S.impact_params(sample, setup)


def _impact_fields(nx, ny, nz, rng, setup, lam, amp=0.03):
    x, y, z = _axes(nx, ny, nz)
    R = setup.radius
    c = ((nx - 1) / 2.0 + rng.uniform(-2, 2), (ny - 1) / 2.0 + rng.uniform(-2, 2), setup.gap + R)
    inside = (x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2 <= R * R
    rR, rB = _two_colours(inside, lam, 1.0)
    u = _waves(nx, ny, nz, rng, amp)
    u[2] -= torch.where(inside, setup.speed, 0.0).float()
    return rR, rB, u


_KEYS = ("rho_in_R", "rho_in_B", "alpha_R", "alpha_B", "tau_R", "tau_B", "tau_e", "tau_q",
         "tau_pi", "A_R", "A_B", "beta", "delta", "ref_R", "ref_B", "contact_angle_deg")


def _plain(p):
    """lbm_params as the dict the 64-bit reference reads."""
    d = {k: float(getattr(p, k)) for k in _KEYS}
    d.update(nx=p.nx, ny=p.ny, nz=p.nz, wall=tuple(p.wall), force=tuple(p.force),
             gravity=tuple(p.gravity), wetting=p.wetting, bgk=p.collision, improved=p.improved)
    return d


def _scene(case, seed):
    """(lbm_params, rho_R, rho_B, u) of one lattice."""
    rng = np.random.default_rng(seed)
    nx, ny, nz, scene = case["nx"], case["ny"], case["nz"], case["scene"]
    kw = dict(storage=case["storage"], collision=case["collision"])
    if scene == "droplet":  # density ratio 10, sigma 0.005 (the benchmark's droplet)
        pd = dict(P.droplet_case(dict(edge=nx, density_ratio=10.0, sigma=0.005)), ny=ny, nz=nz,
                  ref_B=1.0, **kw)
        return (lbm.make_params(**pd), *_droplet(nx, ny, nz, rng, pd, 0.05))
    if scene == "channel":  # equal densities, viscosity ratio 10, peak speed about 0.05
        h, a = ny / 2.0, ny / 4.0
        tau_R, tau_B = 5.5, 1.0
        g = 0.1 * (tau_B - 0.5) / 3.0 / (h * h)
        p = lbm.make_params(nx, ny, nz, wall=(0, 1, 0), tau_R=tau_R, tau_B=tau_B, A_R=1e-3,
                            A_B=1e-3, force=(g, 0.0, 0.0), ref_B=1.0, **kw)
        _, y, _ = _axes(nx, ny, nz)
        yc = (y + 0.5 - h).expand(nz, ny, nx)
        rR, rB = _two_colours(yc.abs() <= a, 1.0, 1.0)
        u = _waves(nx, ny, nz, rng, 0.002)
        u[0] += (0.05 * (1.0 - (yc / h) ** 2)).float()
        return p, rR, rB, u
    if scene == "rt":
        pd = dict(RT.rt_params(L=nx), ny=ny, nz=nz, **kw)
        p = lbm.make_params(**pd)
        p.ref_R, p.ref_B = pd["rho_in_R"], pd["rho_in_B"]
        x, y, z = _axes(nx, ny, nz)
        px, py = rng.uniform(0, 2 * math.pi, 2)
        mode = torch.cos(2 * math.pi * x / nx + px) + torch.cos(2 * math.pi * y / ny + py)
        zi = nz / 2.0
        rR, rB = _two_colours(z >= zi + 0.05 * nx * mode, pd["rho_in_R"], pd["rho_in_B"])
        u = _waves(nx, ny, nz, rng, 0.01)
        u[2] += (0.02 * mode * torch.exp(-(z - zi).abs() / nx)).float()
        return p, rR, rB, u
    sample = dict(density_ratio=8.0, viscosity_ratio=10.0, weber=40.0, reynolds=60.0,
                  theta_deg=70.0)
    setup, p = _impact_scene(nx, ny, nz, sample)
    p.storage, p.collision = lbm.STORAGE[case["storage"]], lbm.COLLISION[case["collision"]]
    p.wall[0] = p.wall[1] = 1
    return (p, *_impact_fields(nx, ny, nz, rng, setup, sample["density_ratio"]))


def _batch_scene(case, seed):
    """One (lbm_params, rho_R, rho_B, u) per case."""
    rng = np.random.default_rng(seed)
    if case["scene"] == "impacts":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        setup = S.ImpactSetup(radius=8, box=(nx, ny, nz))
        for s in S.sample_impacts(case["ncases"], setup, seed=2024):
            p = S.impact_params(s, setup)
            p.storage = lbm.STORAGE[case["storage"]]
            yield (p, *_impact_fields(nx, ny, nz, rng, setup, s["density_ratio"], 0.003))
    else:
        for s in W.droplet_sweep(case["ncases"]):
            s = dict(s, edge=s["edge"] + case["extra"])
            pd = dict(P.droplet_case(s), storage=case["storage"], ref_B=1.0)
            n = s["edge"]
            yield (lbm.make_params(**pd), *_droplet(n, n, n, rng, pd, 0.01 + 0.4 * s["speed"]))


def _network(case, seed):
    """Inputs in [-1, 1]^5 and smooth standardised targets."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = case["rows"] * case.get("steps", 1)
    X = torch.rand((n, 5), generator=g, device=_dev()) * 2 - 1
    k = torch.arange(1, case["n_out"] + 1, device=_dev(), dtype=torch.float32)[None, :]
    T = torch.sin(X[:, :1] + 0.2 * k) + X[:, 1:2] * torch.cos(0.3 * k * X[:, 2:3]) - X[:, 3:4] * X[:, 4:]
    return X, T.contiguous()


def _weights(case, seed):
    """The flat parameter vector the network starts from, in float32."""
    rng = np.random.default_rng(seed)
    dims = [5] + [case["width"]] * case["depth"] + [case["n_out"]]
    parts = []
    for a, b in zip(dims[:-1], dims[1:]):
        parts += [rng.uniform(-1, 1, a * b) * math.sqrt(6.0 / (a + b)), rng.uniform(-0.1, 0.1, b)]
    return np.concatenate(parts).astype(np.float32), dims


def _dtype(storage):
    return {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[storage]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("predict", "train"):
        X, T = _network(case, seed)
        net = S.Surrogate(case["n_out"], width=case["width"], depth=case["depth"],
                          max_batch=case["rows"], seed=seed)
        theta, _ = _weights(case, seed)
        lbm.lbm_mlp_set_params(net.m, theta)
        if kind == "predict":
            return dict(kind=kind, net=net, X=X)
        b = case["rows"]
        xs = [X[k * b:(k + 1) * b].contiguous() for k in range(case["steps"])]
        ts = [T[k * b:(k + 1) * b].contiguous() for k in range(case["steps"])]
        out = torch.empty(theta.size, dtype=torch.float32, device=_dev())
        torch.cuda.synchronize()
        return dict(kind=kind, net=net, xs=xs, ts=ts, rows=b, theta=out)
    stream = torch.cuda.Stream(_dev())
    if kind == "batch":
        scenes = list(_batch_scene(case, seed))
        ps = [s[0] for s in scenes]
        obj = lbm.Batch(ps, stream=stream)
        for k, s in enumerate(scenes):
            obj.init_fields(k, *s[1:])
        del scenes
        st = dict(kind=kind, obj=obj, ps=ps, steps=case["steps"], storage=case["storage"])
        if case["storage"] == "f32" and case["scene"] == "impacts":
            st["out"] = torch.empty((len(ps), 5) + obj.shapes[0], device=_dev())
        elif case["storage"] == "f32":
            st["out"] = [torch.empty((5,) + shape, device=_dev()) for shape in obj.shapes]
        else:
            st["out"] = torch.empty(lbm.lbm_population_bytes(obj.ctx) // 2,
                                    dtype=_dtype(case["storage"]), device=_dev())
        return st
    p, rR, rB, u = _scene(case, seed)
    obj = (lbm.InPlaceLattice if kind == "inplace" else lbm.Lattice)(p, stream=stream)
    obj.init_fields(rR, rB, u)
    st = dict(kind=kind, obj=obj, steps=case["steps"], read=case.get("read"),
              storage=case["storage"], N=p.nx * p.ny * p.nz)
    if case.get("read") == "checkpoint":
        st["out"] = torch.empty(lbm.lbm_population_bytes(obj.ctx) // 2,
                                dtype=_dtype(case["storage"]), device=_dev())
    return st


def _pairs(flat, N):
    """The [direction][cell][colour] values of a raw checkpoint (planes are padded to 64 cells)."""
    plane = (N + 63) // 64 * 64
    return flat[:19 * plane * 2].view(19, plane, 2)[:, :N]


def run(st):
    kind = st["kind"]
    if kind == "predict":
        return st["net"].predict_device(st["X"])
    if kind == "train":
        net = st["net"]
        loss = None
        with torch.cuda.stream(net.stream):
            for k, (x, t) in enumerate(zip(st["xs"], st["ts"])):
                loss = lbm.lbm_mlp_train_step(net.m, x, t, st["rows"], 1e-3,
                                              want_loss=k == len(st["xs"]) - 1)
            lbm.lbm_mlp_get_params(net.m, st["theta"])
        return {"loss": loss, "theta": st["theta"]}
    obj = st["obj"]
    obj.step(st["steps"])
    if kind == "batch":
        if st["storage"] == "f32":
            for k, o in enumerate(st["out"]):
                lbm.lbm_batch_moments(obj.ctx, k, o[0], o[1], o[2:])
            lbm.lbm_sync(obj.ctx)
            return st["out"]
        lbm.lbm_get_populations(obj.ctx, st["out"])
        return _split(st["out"], st["ps"])
    if kind == "inplace":
        if st["storage"] != "f32":
            return {"f": obj.f}
        rR, rB, u = obj.moments()
        return {"rho_R": rR, "rho_B": rB, "u": u, "f": obj.f}
    if st["read"] == "checkpoint":
        lbm.lbm_get_populations(obj.ctx, st["out"])
        return {"state": _pairs(st["out"], st["N"])}
    rR, rB, u = obj.moments()
    out = {"rho_R": rR, "rho_B": rB, "u": u}
    if st["read"] == "state":
        out["f"] = obj.get_f()
    return out


def _split(flat, ps):
    at, out = 0, []
    for p in ps:
        N = p.nx * p.ny * p.nz
        out.append(_pairs(flat[at:], N))
        at += 2 * 19 * ((N + 63) // 64 * 64)
    return out


def work(case):
    kind = case["kind"]
    if kind in ("predict", "train"):
        dims = [5] + [case["width"]] * case["depth"] + [case["n_out"]]
        mac = sum(a * b for a, b in zip(dims[:-1], dims[1:]))
        par = mac + sum(dims[1:])
        if kind == "predict":
            return {"bytes": 4.0 * (case["rows"] * (5 + case["n_out"]) + par),
                    "flops": 2.0 * mac * case["rows"]}
        n = case["steps"]  # theta and both Adam moments read and written, x and t read
        return {"bytes": n * 4.0 * (6 * par + case["rows"] * (5 + case["n_out"])),
                "flops": n * 6.0 * mac * case["rows"]}
    if kind == "batch":
        if case["scene"] == "impacts":
            cells = case["ncases"] * case["nx"] * case["ny"] * case["nz"]
        else:
            cells = sum((s["edge"] + case["extra"]) ** 3 for s in W.droplet_sweep(case["ncases"]))
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
    pop = 38 * (4 if case["storage"] == "f32" else 2)  # 19 directions of two colours
    per = 2.0 * pop * case["steps"]
    if case["storage"] != "f32":
        per += 0 if kind == "inplace" else 2 * pop
    else:
        per += pop + 20
        if case.get("read") == "state":
            per += 2 * pop
    return {"bytes": per * cells, "flops": 700.0 * cells * case["steps"]}


# ---------------------------------------------------------------------------
# The same computation in 64 bits, in plain torch
# ---------------------------------------------------------------------------
_E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
      (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]
_DIM = (2, 1, 0)  # tensor dimension of the x, y and z axis


def _M():
    rows = [lambda x, y, z: 1, lambda x, y, z: x, lambda x, y, z: y, lambda x, y, z: z,
            lambda x, y, z: x * x + y * y + z * z, lambda x, y, z: 2 * x * x - y * y - z * z,
            lambda x, y, z: y * y - z * z, lambda x, y, z: x * y, lambda x, y, z: x * z,
            lambda x, y, z: y * z, lambda x, y, z: x * x * y, lambda x, y, z: x * y * y,
            lambda x, y, z: x * x * z, lambda x, y, z: x * z * z, lambda x, y, z: y * y * z,
            lambda x, y, z: y * z * z, lambda x, y, z: x * x * y * y, lambda x, y, z: x * x * z * z,
            lambda x, y, z: y * y * z * z]
    return np.array([[r(*e) for e in _E] for r in rows], dtype=np.float64)


def _apply(A, f):
    out = []
    for row in A:
        acc = None
        for c, v in zip(row, f):
            if c != 0:
                acc = (v * float(c) if acc is None else acc.add_(v, alpha=float(c)))
        out.append(acc if acc is not None else torch.zeros_like(f[0]))
    return out


def _neighbour(psi, e, wall):
    """psi(x + e); beyond a wall the cell's own value."""
    r = torch.roll(psi, [-e[0], -e[1], -e[2]], [2, 1, 0])
    for a in range(3):
        if e[a] and wall[a]:
            k = psi.shape[_DIM[a]] - 1 if e[a] > 0 else 0
            r.select(_DIM[a], k).copy_(psi.select(_DIM[a], k))
    return r


def _gradient(psi, wall, axes=(0, 1, 2)):
    g = {a: torch.zeros_like(psi) for a in axes}
    for i in range(1, 19, 2):
        e = _E[i]
        if not any(e[a] for a in axes):
            continue
        d = _neighbour(psi, e, wall) - _neighbour(psi, [-v for v in e], wall)
        w = 1.0 / 6.0 if i <= 6 else 1.0 / 12.0
        for a in axes:
            if e[a]:
                g[a].add_(d, alpha=e[a] * w)
    return [g[a] for a in axes]


def _wet(d, G):
    """The contact-angle rule at cells next to a wall."""
    like = G[0]
    n = []
    for a, size in enumerate((d["nx"], d["ny"], d["nz"])):
        v = torch.zeros(size, dtype=like.dtype, device=like.device)
        if d["wall"][a]:
            v[0] += 1.0
            v[-1] -= 1.0
        shape = [1, 1, 1]
        shape[_DIM[a]] = size
        n.append(v.view(shape).expand_as(like))
    nn = n[0] ** 2 + n[1] ** 2 + n[2] ** 2
    s = 1.0 / nn.clamp(min=1.0).sqrt()
    n = [v * s for v in n]
    gn = sum(g * v for g, v in zip(G, n))
    t = [g - gn * v for g, v in zip(G, n)]
    tt, g2 = sum(v * v for v in t), sum(v * v for v in G)
    act = (nn > 0) & (tt > 0) & (g2 > 0)
    th = math.radians(d["contact_angle_deg"])
    it, gm = 1.0 / tt.clamp(min=1e-300).sqrt(), g2.sqrt()
    return [torch.where(act, gm * (-math.cos(th) * v + math.sin(th) * w * it), g)
            for v, w, g in zip(n, t, G)]


def _meq(rho, p, pc, u):
    """Moments 0-18 of the equilibrium of total density rho and pressure p."""
    x, y, z = u
    x2, y2, z2 = x * x, y * y, z * z
    return [rho, rho * x, rho * y, rho * z, 3 * p + rho * (x2 + y2 + z2),
            rho * (2 * x2 - y2 - z2), rho * (y2 - z2), rho * x * y, rho * x * z, rho * y * z,
            pc * y, pc * x, pc * z, pc * x, pc * z, pc * y,
            (2 * p + rho * (2 * x2 + 2 * y2 - z2)) / 6, (2 * p + rho * (2 * x2 + 2 * z2 - y2)) / 6,
            (2 * p + rho * (2 * y2 + 2 * z2 - x2)) / 6]


def _equilibrium(d, rho, alpha, u):
    p = rho * (0.5 * (1.0 - alpha))
    return _apply(np.linalg.inv(_M()), _meq(rho, p, p if d["improved"] else rho / 3.0, u))


def _macro(d, f):
    rR, rB = sum(f[0]), sum(f[1])
    rho = rR + rB
    u = []
    for a in range(3):
        j = sum((f[0][i] + f[1][i]) * float(_E[i][a]) for i in range(19) if _E[i][a])
        u.append((j + 0.5 * (d["force"][a] + rho * d["gravity"][a])) / rho)
    return rR, rB, u


def _collide(d, f):
    """Post-recolouring populations of both colours (lists of 19 fields)."""
    M, wall = _M(), d["wall"]
    cs = [0.5 * (1 - d["alpha_R"]), 0.5 * (1 - d["alpha_B"])]
    rR, rB, u = _macro(d, f)
    rho = rR + rB
    rn = (rR / d["rho_in_R"] - rB / d["rho_in_B"]) / (rR / d["rho_in_R"] + rB / d["rho_in_B"])
    q = rR * (1 - 3 * cs[0]) + rB * (1 - 3 * cs[1])
    G = _gradient(rn, wall)
    Q = [_gradient(u[a] * q, wall, (a,))[0] for a in range(3)] if d["improved"] else None
    if d["wetting"] and any(wall):
        G = _wet(d, G)
    tR, tB, dl = d["tau_R"], d["tau_B"], d["delta"]
    th = 2 * tR * tB / (tR + tB)
    sa, sb = 2 * (tR - th) / dl, 2 * (th - tB) / dl
    tau = torch.where(rn > 0, th + sa * rn - sa / (2 * dl) * rn * rn,
                      th + sb * rn + sb / (2 * dl) * rn * rn)
    tau = torch.where(rn > dl, tR, torch.where(rn < -dl, tB, tau))
    sv = 1.0 / tau
    se, sq, sp = (sv,) * 3 if d["bgk"] else tuple(1.0 / d[k] for k in ("tau_e", "tau_q", "tau_pi"))
    rate = {4: se, 16: sp, 17: sp, 18: sp}
    rate.update({r: sv for r in range(5, 10)})
    rate.update({r: sq for r in range(10, 16)})
    p = rR * cs[0] + rB * cs[1]
    f = [a + b for a, b in zip(*f)]
    m = _apply(M[4:], f)
    eq = _meq(rho, p, p if d["improved"] else rho / 3.0, u)[4:]
    F = [d["force"][a] + rho * d["gravity"][a] for a in range(3)]
    x, y, z = (F[a] * u[a] for a in range(3))
    src = [2 * (x + y + z), 2 * (2 * x - y - z), 2 * (y - z), F[0] * u[1] + F[1] * u[0],
           F[0] * u[2] + F[2] * u[0], F[1] * u[2] + F[2] * u[1], F[1] / 3, F[0] / 3, F[2] / 3,
           F[0] / 3, F[2] / 3, F[1] / 3, (2 * x + 2 * y - z) / 3, (2 * x + 2 * z - y) / 3,
           (2 * y + 2 * z - x) / 3]
    if d["improved"]:
        src[0] = src[0] + Q[0] + Q[1] + Q[2]
        src[1] = src[1] + 2 * Q[0] - Q[1] - Q[2]
        src[2] = src[2] + Q[1] - Q[2]
    g2 = G[0] ** 2 + G[1] ** 2 + G[2] ** 2
    gm = g2.sqrt()
    n = [torch.where(gm >= 1e-12, g / gm.clamp(min=1e-300), 0.0) for g in G]
    A = 0.5 * (d["A_R"] + d["A_B"]) * gm
    x2, y2, z2 = (v * v for v in n)
    pert = {4: -4.0 / 9 * A * (x2 + y2 + z2), 5: 2.0 / 9 * A * (2 * x2 - y2 - z2),
            6: 2.0 / 9 * A * (y2 - z2), 7: 2.0 / 9 * A * n[0] * n[1], 8: 2.0 / 9 * A * n[0] * n[2],
            9: 2.0 / 9 * A * n[1] * n[2], 16: -A * z2 / 9, 17: -A * y2 / 9, 18: -A * x2 / 9}
    dm = [torch.zeros_like(rho)] + [F[a] if torch.is_tensor(F[a]) else torch.full_like(rho, F[a])
                                    for a in range(3)]
    for r in range(4, 19):
        s = rate[r]
        v = (eq[r - 4] - m[r - 4]) * s + src[r - 4] * (1 - 0.5 * s)
        dm.append(v + pert[r] * s if r in pert else v)
    del m, eq, src, pert
    fs = [a.add_(b) for a, b in zip(f, _apply(np.linalg.inv(M).round(12), dm))]
    del dm
    wR, wB = rR / rho, rB / rho
    cb = d["beta"] * wR * wB * p
    out = [[], []]
    for i in range(19):
        l2 = sum(v * v for v in _E[i])
        seg = 0.0
        if i:
            en = sum(n[a] * float(_E[i][a]) for a in range(3) if _E[i][a])
            seg = cb * en * (1.0 / 6 if l2 == 1 else 1.0 / (12 * math.sqrt(2.0)))
        out[0].append(wR * fs[i] + seg)
        out[1].append(wB * fs[i] - seg)
        fs[i] = None
    return out


def _stream(d, fp):
    out = []
    for c in fp:
        new = []
        for i in range(19):
            e = _E[i]
            r = torch.roll(c[i], list(e), [2, 1, 0])
            for a in range(3):
                if e[a] and d["wall"][a]:
                    k = 0 if e[a] > 0 else r.shape[_DIM[a]] - 1
                    r.select(_DIM[a], k).copy_(c[_OPP[i]].select(_DIM[a], k))
            new.append(r)
        out.append(new)
    return out


def _simulate(p, rR, rB, u, steps):
    """(parameters, populations after the last streaming, before it) in 64 bits."""
    d = _plain(p)
    uu = [u[a].double() for a in range(3)]
    f = [_equilibrium(d, rR.double(), d["alpha_R"], uu),
         _equilibrium(d, rB.double(), d["alpha_B"], uu)]
    fp = None
    for _ in range(steps):
        fp = None
        fp = _collide(d, f)
        f = None
        f = _stream(d, fp)
    return d, f, fp


def _deviation(d, f, storage):
    """Stored values: f, or its deviation from each colour's reference rest state."""
    if storage == "f32":
        return f
    for c, (ref, al) in enumerate(((d["ref_R"], d["alpha_R"]), (d["ref_B"], d["alpha_B"]))):
        for i in range(19):
            l2 = sum(v * v for v in _E[i])
            f[c][i] -= ref * (al if l2 == 0 else (1 - al) / (12 if l2 == 1 else 24))
    return f


def _checkpoint(d, fp, storage):
    fp = _deviation(d, fp, storage)
    return torch.stack([torch.stack([fp[0][i].reshape(-1), fp[1][i].reshape(-1)], -1)
                        for i in range(19)])


def _exact_network(case, seed):
    X, T = (v.double() for v in _network(case, seed))
    theta, dims = _weights(case, seed)
    th = torch.as_tensor(theta, dtype=torch.float64, device=_dev())

    def layers(t):
        out, at = [], 0
        for a, b in zip(dims[:-1], dims[1:]):
            out.append((t[at:at + a * b].view(a, b), t[at + a * b:at + a * b + b]))
            at += a * b + b
        return out

    def forward(t, x):
        ls = layers(t)
        for k, (w, b) in enumerate(ls):
            x = x @ w + b
            if k < len(ls) - 1:
                x = torch.tanh(x)
        return x

    if case["kind"] == "predict":
        return forward(th, X)
    m, v, loss, rows = torch.zeros_like(th), torch.zeros_like(th), None, case["rows"]
    for k in range(case["steps"]):
        th = th.detach().requires_grad_(True)
        loss = ((forward(th, X[k * rows:(k + 1) * rows]) - T[k * rows:(k + 1) * rows]) ** 2).mean()
        (g,) = torch.autograd.grad(loss, th)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        mh, vh = m / (1 - 0.9 ** (k + 1)), v / (1 - 0.999 ** (k + 1))
        th = th.detach() - 1e-3 * mh / (vh.sqrt() + 1e-8)
    return {"loss": float(loss.detach()), "theta": th}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("predict", "train"):
        return _exact_network(case, seed)
    if kind == "batch":
        outs = []
        for p, rR, rB, u in _batch_scene(case, seed):
            d, f, fp = _simulate(p, rR, rB, u, case["steps"])
            if case["storage"] == "f32":
                a, b, v = _macro(d, f)
                outs.append(torch.stack([a, b] + v))
            else:
                outs.append(_checkpoint(d, fp, case["storage"]))
        return torch.stack(outs) if case["storage"] == "f32" and case["scene"] == "impacts" else outs
    p, rR, rB, u = _scene(case, seed)
    d, f, fp = _simulate(p, rR, rB, u, case["steps"])
    if kind == "inplace":
        # an even number of steps: the population array is f(x, t) itself
        a, b, v = _macro(d, f)
        fields = {"rho_R": a, "rho_B": b, "u": torch.stack(v)}
        del fp
        state = {"f": torch.stack([torch.stack(c) for c in _deviation(d, f, case["storage"])])}
        return dict(fields, **state) if case["storage"] == "f32" else state
    if case["read"] == "checkpoint":
        del f
        return {"state": _checkpoint(d, fp, case["storage"])}
    a, b, v = _macro(d, f)
    out = {"rho_R": a, "rho_B": b, "u": torch.stack(v)}
    if case["read"] == "state":
        out["f"] = torch.stack([torch.stack(c) for c in f])
    return out

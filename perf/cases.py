"""The workloads whose speed this framework is held to.

Each case is one piece of work that a user of the library has it do, through
the public entry points of ``paper_2204_03775_gb300``, from the arrays that the
user has in hand to the arrays that the user takes away:

* ``shot``      one source gather from rest: the fields zeroed, the source and
                the receivers placed, nt steps, the traces and the final state
                taken out. ``host`` cases take numpy arrays, as a small script
                does; the others stay on the GPU.
* ``resume``    a saved state (u, u_prev) put back, n steps, the state and the
                traces taken out again: checkpoint/restart, and a long run seen
                a few steps at a time. In FP32, FP16 or BF16 field storage.
* ``batch``     many shots on uneven grids, advanced together.
* ``gradient``  the summed misfit gradient of several shots
                (``ws_adjoint_gradient_shots``): one iteration of an inversion.
* ``autograd``  the torch function of one shot's traces, forward and backward,
                in a new model, as an optimizer steps it.
* ``monitor``   a new model and state, the discrete energy before and after a
                few steps (the conservation check of a run), through
                ``ws_energy`` and ``ws_energy_noalloc``.

Sizes are those of the repository's tests and benchmark (64^3 cube, 101x37x45,
256^3, 512^3 and 1024^3 surveys, batches of 96 to 320 cells a side) and the
755 x 994 x 1000 grid of the paper's experiments.
"""

import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2204_03775_gb300 as wsb
from paper_2204_03775_gb300 import autograd as wsa

H = 10.0            # grid spacing, m
CFL = 0.4           # max(V) dt / h
VMIN, VMAX = 1500.0, 4500.0
C = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)
STORAGE = {"fp32": wsb.WS_STORAGE_FP32, "fp16": wsb.WS_STORAGE_FP16, "bf16": wsb.WS_STORAGE_BF16}


def _case(name, kind, nx, ny, nz, steps, rec=8, nb=0, a=0.015, nsrc=1, storage="fp32", host=False,
          nshots=1):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "steps": steps, "rec": rec, "nb": nb, "a": a,
         "nsrc": nsrc, "storage": storage, "host": host, "nshots": nshots}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest whole run: the homogeneous cube, every step a few
        # microseconds of work, so launches and latency count
        _case("cube64_shot", "shot", 64, 64, 64, 100, rec=4),
        # a small script with numpy arrays: a grid ragged in x, y and z, taper,
        # two sources
        _case("ragged101_shot_host", "shot", 101, 37, 45, 60, rec=5, nb=8, a=0.05, nsrc=2, host=True),
        # the smallest call: a saved state, one step, the state out again
        _case("restart96_one_step", "resume", 96, 80, 72, 1, rec=4, nb=16, a=0.02),
        # the survey at the size of one inversion shot (fields near L2's size)
        _case("survey256", "resume", 256, 256, 256, 200, rec=32, nb=20),
        # the benchmark's survey at full size
        _case("survey1024", "resume", 1024, 1024, 1024, 60, rec=32, nb=20),
        # the grid of the paper's experiments: ragged rows and tiles, large
        _case("paper755x994x1000", "resume", 755, 994, 1000, 20, rec=32, nb=20),
        # 16-bit field storage on a survey, and on a smaller ragged grid
        _case("fp16_survey512", "resume", 512, 512, 512, 100, rec=32, nb=20, storage="fp16"),
        _case("bf16_ragged", "resume", 320, 217, 181, 60, rec=16, nb=16, a=0.02, storage="bf16"),
        # uneven shots on one GPU
        _case("batch32", "batch", 320, 320, 256, 60, rec=8, nb=16, a=0.02, nshots=32),
        # inversion: the gradient of several shots in one call, and one shot
        # through torch
        _case("gradient4", "gradient", 192, 160, 144, 64, rec=32, nb=16, a=0.02, nshots=4),
        _case("autograd128", "autograd", 128, 128, 128, 49, rec=24, nb=16, a=0.02),
        # model update and energy check
        _case("monitor_energy", "monitor", 320, 288, 256, 8, rec=0),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["shot", "shot", "resume", "resume", "resume16", "batch", "gradient",
                       "autograd", "monitor"])
    nb = rng.choice([0, 8, 16, 20])
    a = rng.choice([0.015, 0.02, 0.05])
    if kind == "shot":
        return _case(None, kind, size(33, 200), size(24, 200), size(20, 200), size(40, 120),
                     rec=rng.choice([1, 4, 8]), nb=min(nb, 8), a=a, nsrc=rng.choice([1, 2, 5]),
                     host=rng.random() < 0.3)
    if kind == "resume":
        return _case(None, kind, size(64, 900), size(48, 900), size(40, 900), size(1, 40),
                     rec=rng.choice([4, 16, 32]), nb=nb, a=a)
    if kind == "resume16":
        return _case(None, "resume", size(64, 640), size(24, 640), size(30, 640), size(1, 60),
                     rec=rng.choice([4, 16]), nb=nb, a=a, storage=rng.choice(["fp16", "bf16"]))
    if kind == "batch":    # the sizes given are the largest of each axis
        return _case(None, kind, rng.randint(128, 320), rng.randint(128, 320), rng.randint(128, 256),
                     rng.randint(20, 60), rec=8, nb=min(nb, 16), a=a, nshots=rng.randint(2, 32))
    if kind == "gradient":
        return _case(None, kind, size(64, 200), size(48, 200), size(48, 160), size(36, 64),
                     rec=rng.choice([8, 16, 32]), nb=min(nb, 16), a=a, nshots=rng.randint(1, 6))
    if kind == "autograd":
        return _case(None, kind, size(48, 180), size(40, 180), size(40, 180), size(36, 64),
                     rec=rng.choice([8, 16, 24]), nb=min(nb, 16), a=a)
    return _case(None, "monitor", size(40, 400), size(40, 400), size(40, 300), size(1, 8), rec=0)


# ------------------------------------------------------------------ inputs


def _gen(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * seed + tag)
    return g


def _smooth(shape, seed, tag, spacing):
    """Smooth random field in [-1, 1]: coarse noise, trilinear upsampling."""
    coarse = tuple(max(2, -(-n // spacing) + 1) for n in shape)
    t = torch.randn((1, 1) + coarse, generator=_gen(seed, tag), device="cuda")
    t /= t.abs().max()
    size = tuple((m - 1) * spacing + 1 for m in coarse)
    t = F.interpolate(t, size=size, mode="trilinear", align_corners=True)[0, 0]
    nz, ny, nx = shape
    return t[:nz, :ny, :nx].contiguous()


def _model(shape, seed, tag=1):
    """Ten layers from 1500 to 4500 m/s with 5 % smooth noise, float32."""
    nz = shape[0]
    layer = torch.clamp(torch.arange(nz, device="cuda") * 10 // nz, max=9).to(torch.float32)
    v = _smooth(shape, seed, tag, 8)
    v *= 0.05
    v += 1.0
    v *= (VMIN + layer * ((VMAX - VMIN) / 9.0))[:, None, None]
    return v.clamp_(VMIN, VMAX)


def _cube_model(shape):
    return torch.full(shape, 2000.0, device="cuda")


def _wavefield(shape, seed, tag):
    """A wavefield everywhere in the grid: u and the level before it."""
    u = _smooth(shape, seed, tag, 6)
    p = _smooth(shape, seed, tag + 1, 6)
    p *= 0.2
    p += u
    return u, p


def _cube(case):
    """The homogeneous cube: the one workload without layers and noise."""
    return case["kind"] == "shot" and case["nx"] == case["ny"] == case["nz"] and case["nb"] == 0


def _dt(case):
    return CFL * H / (2000.0 if _cube(case) else VMAX)


def _plane(kind):
    """The receivers' plane of each kind of run."""
    return {"shot": 0, "resume": 20, "batch": 16, "gradient": 6, "autograd": 6, "monitor": 0}[kind]


def _receivers(nx, ny, nz, side, plane):
    """side x side on a plane, evenly spread (all the way to the last cell)."""
    k = min(plane, nz - 1)
    ii = [min(nx - 1, int((p + 0.5) * nx / side)) for p in range(side)]
    jj = [min(ny - 1, int((q + 0.5) * ny / side)) for q in range(side)]
    r = [[i, j, k] for j in jj for i in ii]
    if side % 2:   # odd sides: some receivers in corners of the grid
        r += [[0, 0, 0], [nx - 1, ny - 1, nz - 1]]
    return np.array(r, dtype=np.int32)


def _sources(case, seed, shot=0):
    """(i, j, k, f0, t0, amp) drawn inside the grid, early enough to radiate."""
    rng = np.random.Generator(np.random.PCG64([seed, shot, 77]))
    dt = _dt(case)
    out = []
    for _ in range(case["nsrc"]):
        cell = [int(rng.integers(n // 4, max(n // 4 + 1, 3 * n // 4)))
                for n in (case["nx"], case["ny"])]
        # the centre of the cube; elsewhere near the receivers' plane, so that
        # the first arrivals fall inside the recording
        cell.append(case["nz"] // 2 if _cube(case)
                    else min(case["nz"] - 1, _plane(case["kind"]) + int(rng.integers(2, 12))))
        f0 = float(rng.uniform(0.6, 1.0) / (25.0 * dt))    # 25 to 40 steps a period
        out.append((cell[0], cell[1], cell[2], f0, 0.8 / f0, float(rng.uniform(0.5, 2.0))))
    return out


def _shape(case):
    return case["nz"], case["ny"], case["nx"]


def _batch_sizes(case):
    rng = np.random.Generator(np.random.PCG64([2204, case["nx"], case["ny"], case["nz"]]))
    return [tuple(int(rng.integers(96, hi + 1)) for hi in (case["nz"], case["ny"], case["nx"]))
            for _ in range(case["nshots"])]


def _handle(case, shape, vel):
    nz, ny, nx = shape
    h = wsb.ws_create(nx, ny, nz, H, _dt(case))
    wsb.ws_set_velocity(h, vel)
    if case["nb"]:
        wsb.ws_set_sponge(h, case["nb"], case["a"])
    if case["storage"] != "fp32":
        wsb.ws_set_storage(h, STORAGE[case["storage"]])
    return h


def _empty(shape):
    return torch.empty(shape, dtype=torch.float32, device="cuda")


def _observed(case, seed):
    """Observed traces of each shot: those of a model 4 % faster in a blob."""
    shape = _shape(case)
    rec = _receivers(case["nx"], case["ny"], case["nz"], case["rec"], _plane(case["kind"]))
    vel = _true_model(case, seed)
    out = []
    for q in range(case["nshots"]):
        tr, _, _ = _run64(vel, case, None, _sources(case, seed, q), rec, case["steps"])
        out.append(tr.to(torch.float32))
    return rec, out


def _true_model(case, seed):
    nz, ny, nx = _shape(case)
    v = _model(_shape(case), seed).double()
    k, j, i = (torch.arange(n, device="cuda", dtype=torch.float64) for n in (nz, ny, nx))
    r2 = ((k - nz / 3)[:, None, None] ** 2 + (j - ny / 2)[None, :, None] ** 2
          + (i - nx / 2)[None, None, :] ** 2)
    return (v * (1.0 + 0.04 * torch.exp(-r2 / 800.0))).clamp(max=1.1 * VMAX)


def prepare(case, seed):
    kind = case["kind"]
    shape = _shape(case)
    nz, ny, nx = shape
    if kind in ("shot", "resume"):
        vel = _cube_model(shape) if _cube(case) else _model(shape, seed)
        h = _handle(case, shape, vel)
        rec = _receivers(nx, ny, nz, case["rec"], _plane(kind))
        s = {"case": case, "h": h, "rec": rec, "src": _sources(case, seed)}
        if kind == "resume":
            s["u"], s["p"] = _wavefield(shape, seed, 11)
            for q in s["src"]:
                wsb.ws_add_source(h, *q)
        if not case["host"]:
            s["traces"] = _empty((len(rec), case["steps"]))
            s["out"] = _empty(shape), _empty(shape)
        return s
    if kind == "batch":
        sizes = _batch_sizes(case)
        cells = [z * y * x for z, y, x in sizes]
        flat = [_empty((sum(cells),)) for _ in range(4)]     # u, u_prev in; u, u_prev out
        views = [[] for _ in range(4)]
        at = 0
        shots, recs = [], []
        for q, (sh, n) in enumerate(zip(sizes, cells)):
            for f, v in zip(flat, views):
                v.append(f[at:at + n].view(sh))
            at += n
            u, p = _wavefield(sh, seed, 100 + 4 * q)
            views[0][q].copy_(u)
            views[1][q].copy_(p)
            h = _handle(case, sh, _model(sh, seed, 102 + 4 * q))
            c = dict(case, nz=sh[0], ny=sh[1], nx=sh[2])
            for r in _sources(c, seed, q):
                wsb.ws_add_source(h, *r)
            shots.append(h)
            recs.append(_receivers(sh[2], sh[1], sh[0], case["rec"], _plane(kind)))
        traces = _empty((len(sizes), len(recs[0]), case["steps"]))
        s = {"case": case, "shots": shots, "recs": recs, "views": views, "flat": flat,
             "traces": traces, "batch": wsb.ws_batch_create(shots)}
        wsb.ws_batch_step(s["batch"], 48)     # the batch's own tuning, on real steps
        wsb.ws_batch_synchronize(s["batch"])
        return s
    if kind == "gradient":
        rec, obs = _observed(case, seed)
        vel = _model(shape, seed)
        shots, streams = [], []
        for q in range(case["nshots"]):
            h = _handle(case, shape, vel)
            streams.append(torch.cuda.Stream())
            wsb.ws_set_stream(h, streams[-1])
            for r in _sources(case, seed, q):
                wsb.ws_add_source(h, *r)
            wsb.ws_set_receivers(h, rec, case["steps"])
            shots.append(h)
        return {"case": case, "shots": shots, "streams": streams, "data": obs, "grad": _empty(shape)}
    if kind == "autograd":
        rec, obs = _observed(case, seed)
        m = _model(shape, seed).double().pow_(-2).to(torch.float32)
        shot = wsa.Shot(shape, H, _dt(case), case["steps"], _sources(case, seed), rec,
                        sponge=(case["nb"], case["a"]))
        return {"case": case, "shot": shot, "m": m, "obs": obs[0]}
    u, p = _wavefield(shape, seed, 11)
    vel = _model(shape, seed)
    return {"case": case, "h": _handle(case, shape, vel), "vel": vel, "u": u, "p": p,
            "e": torch.zeros(1, dtype=torch.float64, device="cuda"),
            "out": (_empty(shape), _empty(shape))}


# ------------------------------------------------------------------ one pass


def run(state):
    case = state["case"]
    kind, steps = case["kind"], case["steps"]
    if kind == "shot":
        h = state["h"]
        wsb.ws_write_field(h, None, None, 0)
        wsb.ws_clear_sources(h)
        for q in state["src"]:
            wsb.ws_add_source(h, *q)
        wsb.ws_set_receivers(h, state["rec"], steps)
        wsb.ws_step(h, steps)
        if case["host"]:
            traces = wsb.ws_read_traces(h)
            u, p = wsb.ws_read_field(h)
            return {"traces": traces, "u": u, "u_prev": p}
        wsb.ws_read_traces(h, state["traces"])
        u, p = wsb.ws_read_field(h, *state["out"])
        return {"traces": state["traces"], "u": u, "u_prev": p}
    if kind == "resume":
        h = state["h"]
        wsb.ws_write_field(h, state["u"], state["p"], 3)
        wsb.ws_set_receivers(h, state["rec"], steps)
        wsb.ws_step(h, steps)
        wsb.ws_read_traces(h, state["traces"])
        u, p = wsb.ws_read_field(h, *state["out"])
        return {"traces": state["traces"], "u": u, "u_prev": p}
    if kind == "batch":
        ins, inp, outs, outp = state["views"]
        for q, h in enumerate(state["shots"]):
            wsb.ws_write_field(h, ins[q], inp[q], 3)
            wsb.ws_set_receivers(h, state["recs"][q], steps)
        wsb.ws_batch_step(state["batch"], steps)
        for q, h in enumerate(state["shots"]):
            wsb.ws_read_traces(h, state["traces"][q])
            wsb.ws_read_field(h, outs[q], outp[q])
        return {"traces": state["traces"], "u": state["flat"][2], "u_prev": state["flat"][3]}
    if kind == "gradient":
        g, j, norm = wsb.ws_adjoint_gradient_shots(state["shots"], state["data"], wsb.WS_ADJ_DATA,
                                                   state["grad"])
        return {"grad": g, "misfit": j, "norm": norm}
    if kind == "autograd":
        m = state["m"].clone().requires_grad_(True)
        t = wsa.traces(m, state["shot"])
        loss = 0.5 * (t - state["obs"]).square().sum()
        loss.backward()
        return {"traces": t.detach(), "grad": m.grad}
    h = state["h"]
    wsb.ws_set_velocity(h, state["vel"])
    wsb.ws_write_field(h, state["u"], state["p"], 0)
    e0 = wsb.ws_energy(h)
    wsb.ws_step(h, steps)
    e1 = wsb.ws_energy(h)
    u, p = wsb.ws_read_field(h, *state["out"])
    wsb.ws_energy_noalloc(u, p, state["vel"], H, _dt(case), state["e"])
    return {"before": e0, "after": e1, "dense": state["e"], "u": u, "u_prev": p}


# ------------------------------------------------------------------ work


def work(case):
    """Bytes and operations that no implementation of the calls can do without.

    A step is one sweep over the grid: both levels and the model read once,
    one level written once (16 bytes a cell; 10 in 16-bit storage), 51 flops a
    cell as the paper counts them. States that come in or go out are read or
    written once. A gradient needs the forward run, each state once more for
    the imaging (it is stored once and read once, or recomputed at no less),
    the backward run, and its own array.
    """
    n, steps = case["nx"] * case["ny"] * case["nz"], case["steps"]
    kind = case["kind"]
    step = 16.0 if case["storage"] == "fp32" else 10.0
    if kind == "shot":
        return {"bytes": n * (step * steps + 8.0), "flops": 51.0 * n * steps}
    if kind == "resume":
        return {"bytes": n * (step * steps + 16.0), "flops": 51.0 * n * steps}
    if kind == "batch":
        n = sum(z * y * x for z, y, x in _batch_sizes(case))
        return {"bytes": n * (step * steps + 16.0), "flops": 51.0 * n * steps}
    if kind == "gradient":
        return {"bytes": case["nshots"] * n * (40.0 * steps) + 4.0 * n,
                "flops": case["nshots"] * 104.0 * n * steps}
    if kind == "autograd":
        return {"bytes": n * (40.0 * steps + 8.0), "flops": 104.0 * n * steps}
    # monitor: the model in, the state in and out, three energies of 12 bytes
    return {"bytes": n * (step * steps + 4.0 + 16.0 + 36.0), "flops": n * (51.0 * steps + 3 * 60.0)}


# ------------------------------------------------------------------ in 64 bits


def _lap(u, out):
    """h^2 times the 25-point Laplacian, zero outside the grid, into out."""
    torch.mul(u, 3.0 * C[0], out=out)
    for d in range(3):
        n = u.shape[d]
        for m in range(1, 5):
            if n > m:
                out.narrow(d, m, n - m).add_(u.narrow(d, 0, n - m), alpha=C[m])
                out.narrow(d, 0, n - m).add_(u.narrow(d, m, n - m), alpha=C[m])
    return out


def _taper(n, nb, a):
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    d = torch.minimum(i, n - 1 - i)
    return torch.where(d < nb, torch.exp(-(a * (nb - d)) ** 2), torch.ones_like(d))


def _ricker(t, f0, t0, amp):
    x = (math.pi * f0 * (t - t0)) ** 2
    return amp * (1.0 - 2.0 * x) * math.exp(-x)


def _run64(vel, case, state, sources, rec, steps, step0=0, laps=None):
    """(traces, u, u_prev) after `steps` steps of the definition in FP64.

    vel: [nz][ny][nx]; state: (u, u_prev) or None for rest; laps: if a list,
    receives the stencil sum of each step's u."""
    dt = _dt(case)
    nz, ny, nx = vel.shape
    r = (vel.double() * (dt / H)) ** 2
    if state is None:
        u = torch.zeros(vel.shape, dtype=torch.float64, device="cuda")
        p = torch.zeros_like(u)
    else:
        u, p = state[0].double(), state[1].double()
    g = None
    if case["nb"]:
        gx, gy, gz = (_taper(n, case["nb"], case["a"]) for n in (nx, ny, nz))
    tr = torch.zeros((len(rec), steps), dtype=torch.float64, device="cuda")
    ri = torch.as_tensor(np.asarray(rec, dtype=np.int64).reshape(-1, 3), device="cuda")
    lap = torch.empty_like(u)
    for n in range(steps):
        _lap(u, lap)
        if laps is not None:
            laps.append(lap.clone())
        lap.mul_(r)
        lap.add_(u, alpha=2.0)
        if case["nb"]:
            for f in (lap, p):
                f.mul_(gx).mul_(gy[:, None]).mul_(gz[:, None, None])
            # g (2u + W L) - g^2 u_prev
            p.mul_(gx).mul_(gy[:, None]).mul_(gz[:, None, None])
        torch.sub(lap, p, out=p)
        for (i, j, k, f0, t0, amp) in sources:
            p[k, j, i] += r[k, j, i] * (H * H * _ricker((step0 + n) * dt, f0, t0, amp))
        u, p = p, u
        if len(rec):
            tr[:, n] = u[ri[:, 2], ri[:, 1], ri[:, 0]]
    return tr, u, p


def _gradient64(case, vel, sources, rec, obs):
    """(dJ/dm, J, traces) of one shot: the transposed recurrence in FP64."""
    nz, ny, nx = vel.shape
    steps, dt = case["steps"], _dt(case)
    laps = []
    tr, u, p = _run64(vel, case, None, sources, rec, steps, laps=laps)
    del u, p
    res = tr - obs.double()
    v2 = vel.double() ** 2
    w = v2 * (dt / H) ** 2
    g = torch.ones_like(w)
    if case["nb"]:
        for n, shape in ((nx, (1, 1, nx)), (ny, (1, ny, 1)), (nz, (nz, 1, 1))):
            g = g * _taper(n, case["nb"], case["a"]).view(shape)
    ri = torch.as_tensor(np.asarray(rec, dtype=np.int64).reshape(-1, 3), device="cuda")
    at = (ri[:, 2], ri[:, 1], ri[:, 0])
    wg = (w * g)[at]
    r1, r2 = torch.zeros_like(w), torch.zeros_like(w)     # rho^{k+1}, rho^{k+2}
    grad, lap = torch.zeros_like(w), torch.empty_like(w)
    for k in range(steps, 0, -1):
        _lap(r1, lap)
        new = g * (2.0 * r1 - g * r2 + w * lap)
        new.index_put_(at, wg * res[:, k - 1], accumulate=True)
        r1, r2 = new, r1
        grad.addcmul_(r1, laps[k - 1])
        for (i, j, kk, f0, t0, amp) in sources:
            s = H * H * _ricker((k - 1) * dt, f0, t0, amp)
            grad[kk, j, i] += r1[kk, j, i] * s / g[kk, j, i]
    return -v2 * grad, 0.5 * res.square().sum(), tr


def _energy64(vel, case, u, p):
    u, p = u.double(), p.double()
    lap = _lap(p, torch.empty_like(p)).div_(H * H)
    vdt2 = (vel.double() * _dt(case)) ** 2
    return float(((u - p) ** 2 / vdt2 - u * lap).sum())


def exact(case, seed):
    kind, shape = case["kind"], _shape(case)
    nz, ny, nx = shape
    if kind in ("shot", "resume"):
        vel = _cube_model(shape) if _cube(case) else _model(shape, seed)
        rec = _receivers(nx, ny, nz, case["rec"], _plane(kind))
        state = None if kind == "shot" else _wavefield(shape, seed, 11)
        tr, u, p = _run64(vel, case, state, _sources(case, seed), rec, case["steps"],
                          0 if kind == "shot" else 3)
        return {"traces": tr, "u": u, "u_prev": p}
    if kind == "batch":
        trs, us, ps = [], [], []
        for q, sh in enumerate(_batch_sizes(case)):
            c = dict(case, nz=sh[0], ny=sh[1], nx=sh[2])
            tr, u, p = _run64(_model(sh, seed, 102 + 4 * q), c, _wavefield(sh, seed, 100 + 4 * q),
                              _sources(c, seed, q), _receivers(sh[2], sh[1], sh[0], case["rec"], _plane(kind)),
                              case["steps"], 3)
            trs.append(tr)
            us.append(u.reshape(-1))
            ps.append(p.reshape(-1))
        return {"traces": torch.stack(trs), "u": torch.cat(us), "u_prev": torch.cat(ps)}
    if kind in ("gradient", "autograd"):
        rec, obs = _observed(case, seed)
        vel = _model(shape, seed)
        if kind == "autograd":    # the parameter is the float32 squared slowness
            vel = vel.double().pow_(-2).to(torch.float32).double().pow(-0.5)
        total, j, tr = None, 0.0, None
        for q in range(case["nshots"]):
            g, jq, tr = _gradient64(case, vel, _sources(case, seed, q), rec, obs[q])
            total = g if total is None else total + g
            j += float(jq)
        if kind == "autograd":
            return {"traces": tr, "grad": total}
        return {"grad": total, "misfit": j, "norm": float(total.norm())}
    vel = _model(shape, seed)
    u, p = _wavefield(shape, seed, 11)
    none = np.zeros((0, 3), dtype=np.int32)
    _, u1, p1 = _run64(vel, case, (u, p), [], none, case["steps"])
    e1 = _energy64(vel, case, u1, p1)
    return {"before": _energy64(vel, case, u, p), "after": e1, "dense": None, "u": u1, "u_prev": p1}

"""What a program built on this library spends its time on, as cases that can be timed.

A case is a dict of plain values.  `listed()` names the representative ones, `draw(rng)` gives more of the
same ranges, `prepare(case, seed)` makes the inputs (on the GPU) and the model or network a program keeps,
`run(state)` is one pass through the public entry points, `work(case)` the bytes and operations the pass
cannot do without, and `exact(case, seed)` the same outputs in 64 bits by plain torch.

Kinds of case
  run        one source on one velocity model: es_source_set, es_state_reset, es_run, es_state_get
  catalog    a batch of sources sharing one model: es_batch_set, es_run (the surrogate's catalog, the fallback)
  group      batched models of several grid sizes advanced together: es_run_group
  superpose  300-event gathers from single-event traces: es_superpose / es_superpose_noalloc
  predict    the surrogate serving a batch of sources: es_sur_predict
  train      the surrogate's Adam steps: es_sur_train_step, then the parameters
  laplacian  the density Laplacian of the event selection: es_laplacian
"""
import ctypes
import math

import numpy as np
import torch

from paper_1705_04874_gb300 import es, surrogate

VX, VY, VZ, SXX, SYY, SZZ, SXY, SXZ, SYZ = range(9)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _run(name, nx, ny, nz, pml, nt, rx, ry, f0, model="marine", d=(10.0, 10.0, 10.0), tau=0.0, out="device"):
    return {"name": name, "kind": "run", "model": model, "nx": nx, "ny": ny, "nz": nz, "dx": d[0], "dy": d[1],
            "dz": d[2], "pml": pml, "nt": nt, "rx": rx, "ry": ry, "f0": f0, "tau": tau, "out": out}


def listed():
    return [
        # the quick look: a small two-layer box, 16 receivers, traces to the host
        _run("run-32", 32, 32, 32, 6, 300, 4, 4, 25.0, model="layers", out="host"),
        # the everyday marine model
        _run("run-128", 128, 128, 128, 10, 400, 32, 32, 30.0),
        # the largest single-source run
        _run("run-256", 256, 256, 256, 12, 120, 64, 64, 30.0),
        # the paper's own odd grid and spacing, a sensor at every interior x-y point
        _run("run-paper-grid", 125, 75, 301, 10, 200, 105, 55, 30.0, d=(12.5, 12.5, 10.0)),
        # the largest cube the paper fits on one card: no axis a power of two or even smooth
        _run("run-190", 190, 190, 190, 10, 80, 40, 40, 30.0),
        # building the surrogate's catalog: four locations x six unit moment tensors per batch
        {"name": "catalog-96", "kind": "catalog", "n": 96, "pml": 10, "nb": 24, "nt": 128, "rx": 8, "ry": 8,
         "f0": 30.0},
        # many sources on models of three sizes in one graph
        {"name": "group-128-96-160", "kind": "group", "sizes": "128:16,96:4,160:2", "pml": 10, "nt": 64, "rx": 32,
         "ry": 32, "f0": 30.0},
        # a 300-event gather from 64 catalogued sources, everything on the GPU
        {"name": "superpose-300", "kind": "superpose", "n_src": 64, "n_rcv": 1024, "nt": 2000, "events": 300,
         "span": 2.0, "dt": 7.5e-4, "entry": "device"},
        # the smallest call: three events over 16 receivers, host arrays in and out
        {"name": "superpose-3", "kind": "superpose", "n_src": 1, "n_rcv": 16, "nt": 300, "events": 3, "span": 0.05,
         "dt": 1.2e-3, "entry": "host"},
        # the surrogate at its full size, one serving batch
        {"name": "predict-1024", "kind": "predict", "nfreq": 9, "hidden": 768, "latent": 768, "n_rcv": 64, "nt": 1024,
         "batch": 1024},
        # the surrogate at its full size, two training steps
        {"name": "train-256", "kind": "train", "nfreq": 9, "hidden": 768, "latent": 768, "n_rcv": 64, "nt": 1024,
         "batch": 256, "steps": 2},
        # picking event locations on the rock interfaces of the large model
        {"name": "laplacian-256", "kind": "laplacian", "nx": 256, "ny": 256, "nz": 256, "dx": 10.0, "dy": 10.0,
         "dz": 10.0},
    ]


_SMOOTH = (32, 48, 64, 80, 96, 128, 160, 192, 256)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _axis(rng, lo=24, hi=320):
    """An axis length: as often one a user picks for its factors as any other, odd ones among them."""
    return rng.choice([n for n in _SMOOTH if lo <= n <= hi]) if rng.random() < 0.5 else _log(rng, lo, hi)


def _mul8(rng, lo, hi):
    return max(lo, min(hi, 8 * round(_log(rng, lo, hi) / 8)))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "catalog", "group", "superpose", "predict", "train", "laplacian"])
    if kind == "run":
        while True:
            nx, ny, nz = (_axis(rng) for _ in range(3))
            if nx * ny * nz <= 190 ** 3:
                break
        pml = rng.randint(4, min(12, (min(nx, ny, nz) - 12) // 2))
        nt = max(20, min(400, int(5.0e8 / (nx * ny * nz))))
        c = _run("", nx, ny, nz, pml, rng.randint(nt // 2, nt), rng.randint(3, max(3, (nx - 2 * pml) // 2)),
                 rng.randint(3, max(3, (ny - 2 * pml) // 2)), 30.0, d=(10.0, rng.choice([10.0, 12.5]), 10.0),
                 tau=rng.choice([0.0, 0.0, 0.0, 1.0e-4]), out=rng.choice(["device", "host"]))
        del c["name"]
        return c
    if kind == "catalog":
        n = _axis(rng, 40, 160)
        nb = max(2, min(48, int(rng.uniform(0.3, 1.0) * 24 * 96 ** 3 / n ** 3)))
        return {"kind": kind, "n": n, "pml": rng.randint(6, 10), "nb": nb, "nt": rng.randint(30, 90),
                "rx": rng.randint(3, 12), "ry": rng.randint(3, 12), "f0": 30.0}
    if kind == "group":
        sizes = [(n, rng.randint(1, max(1, int(6e6 / n ** 3)))) for n in rng.sample([48, 64, 96, 100, 125, 128], 2)]
        return {"kind": kind, "sizes": ",".join("%d:%d" % s for s in sizes), "pml": rng.randint(6, 10),
                "nt": rng.randint(24, 64), "rx": rng.randint(4, 24), "ry": rng.randint(4, 24), "f0": 30.0}
    if kind == "superpose":
        nt, n_rcv, n_src = _log(rng, 200, 3000), _log(rng, 16, 1024), rng.randint(1, 64)
        return {"kind": kind, "n_src": n_src, "n_rcv": n_rcv, "nt": nt, "events": _log(rng, 2, 300),
                "span": rng.uniform(0.1, 2.0), "dt": rng.uniform(5e-4, 1.5e-3),
                "entry": rng.choice(["device", "noalloc"] if n_src * n_rcv * nt > 4_000_000
                                    else ["device", "noalloc", "host"])}
    if kind in ("predict", "train"):
        c = {"kind": kind, "nfreq": rng.randint(3, 9), "hidden": _mul8(rng, 64, 768), "latent": _mul8(rng, 32, 768),
             "n_rcv": rng.randint(4, 64), "nt": _mul8(rng, 128, 1024), "batch": _mul8(rng, 8, 1024)}
        if kind == "train":
            c.update(batch=min(256, c["batch"]), steps=2)
        return c
    while True:
        nx, ny, nz = (_axis(rng) for _ in range(3))
        if nx * ny * nz <= 256 ** 3:
            return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "dx": 10.0, "dy": 12.5, "dz": 10.0}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _velocity_model(nx, ny, nz, dz, seed, kind="marine"):
    """(rho, cp, cs) [nz][ny][nx] float32 and the number of water cells: a water column over layered sediments
    with a depth gradient and 5 % correlated perturbations, or water over one rock."""
    nw = int(round(0.19 * nz)) if kind == "marine" else nz // 4
    cp = torch.empty((nz, ny, nx), device="cuda", dtype=torch.float64)
    g = torch.randn((nz, ny, nx), device="cuda", generator=_gen(seed), dtype=torch.float32)
    if kind == "layers":
        # the rock's speeds differ from seed to seed, by a few per cent
        s = 1.0 + 0.02 * float(g.flatten()[0].clamp(-2, 2))
        cp[nw:], rho, cs = 2500.0 * s, torch.full_like(cp, 2200.0), torch.full_like(cp, 1200.0 * s)
    else:
        k = [torch.fft.fftfreq(n, device="cuda") for n in (nz, ny)] + [torch.fft.rfftfreq(nx, device="cuda")]
        r2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
        g = torch.fft.irfftn(torch.fft.rfftn(g) * torch.exp(-(math.pi ** 2) * 64.0 * r2 / 2), s=(nz, ny, nx))
        g = (g - g.mean()) / g.std()
        depth = np.empty(nz)
        for i in range(nw, nz):
            layer = min(4, (i - nw) * 5 // max(1, nz - nw))
            top = nw + layer * (nz - nw) // 5
            depth[i] = min(4000.0, 1800.0 + 500.0 * layer + 0.5 * (i - top) * dz)
        cp[nw:] = torch.tensor(depth[nw:], device="cuda")[:, None, None] * (1 + 0.05 * g[nw:].double())
        rho, cs = 310.0 * cp.clamp(min=1.0) ** 0.25, cp / 1.8
    cp[:nw], rho[:nw], cs[:nw] = 1500.0, 1000.0, 0.0
    return [t.float().contiguous() for t in (rho, cp, cs)] + [nw]


def _ricker(nt, dt, f0):
    a = (math.pi * f0 * (np.arange(nt) * dt - 1.0 / f0)) ** 2
    return ((1 - 2 * a) * np.exp(-a)).astype(np.float32)


def _receivers(nx, ny, pml, nw, rx, ry):
    r = np.empty((rx * ry, 3), np.int32)
    for j in range(ry):
        for i in range(rx):
            r[i + rx * j] = (pml + ((2 * i + 1) * (nx - 2 * pml)) // (2 * rx),
                             pml + ((2 * j + 1) * (ny - 2 * pml)) // (2 * ry), nw - 1)
    return r


def _sources(rs, nb, nx, ny, nz, pml, nw):
    """Cells a few below the seabed, in the middle of the grid, and unit-norm symmetric moment tensors."""
    pos = np.empty((nb, 3), np.int32)
    for a, n in ((0, nx), (1, ny)):
        pos[:, a] = rs.randint(max(pml + 1, n // 4), min(n - pml - 3, max(pml + 1, 3 * n // 4)) + 1, nb)
    top = max(nw + 3, pml + 1)
    pos[:, 2] = rs.randint(top, min(top + 6, nz - 3 - pml) + 1, nb)
    m = rs.standard_normal((nb, 6))
    return pos, m / np.sqrt((m[:, :3] ** 2).sum(1) + 2 * (m[:, 3:] ** 2).sum(1))[:, None]


def _solver_inputs(c, seed, n, nb):
    nx, ny, nz = n
    d = [c.get("dx", 10.0), c.get("dy", 10.0), c.get("dz", 10.0)]
    rho, cp, cs, nw = _velocity_model(nx, ny, nz, d[2], seed, c.get("model", "marine"))
    dt = 0.3 * min(d) / float(cp.max())
    pos, mt = _sources(np.random.RandomState(seed % (1 << 31)), nb, nx, ny, nz, c["pml"], nw)
    return {"rho": rho, "cp": cp, "cs": cs, "d": d, "dt": dt, "pos": pos, "mt": mt, "pml": c["pml"], "nt": c["nt"],
            "w": _ricker(c["nt"], dt, c["f0"]), "rcv": _receivers(nx, ny, c["pml"], nw, c["rx"], c["ry"]),
            "tau": min(c.get("tau", 0.0), 0.15 * dt)}


def _model(i, nb=None):
    m = es.Model(i["rho"], i["cp"], i["cs"], dx=i["d"][0], pml=i["pml"])
    if i["d"][1] != i["d"][0] or i["d"][2] != i["d"][0]:
        m.set_spacing(*i["d"])
    if i["tau"]:
        m.set_viscosity(i["tau"])
    return m


def _sizes(c):
    return [tuple(int(v) for v in s.split(":")) for s in c["sizes"].split(",")]


def _arrivals(shape, nt, g):
    """Traces as a solver run leaves them: silence, an arrival, a decaying coda.  shape + [nt], float32."""
    t = torch.arange(nt, device="cuda", dtype=torch.float32)
    t0 = torch.rand(shape, device="cuda", generator=g) * 0.5 * nt
    amp = torch.randn(shape, device="cuda", generator=g)
    x = torch.randn(tuple(shape) + (nt,), device="cuda", generator=g)
    u = t - t0[..., None]
    return x.mul_(amp[..., None] * torch.exp(-u.clamp(min=0) * (4.0 / nt))).mul_(u >= 0)


def _superpose_inputs(c, seed):
    g, rs = _gen(seed), np.random.RandomState(seed % (1 << 31))
    tr = torch.empty((c["n_src"], 4, c["n_rcv"], c["nt"]), device="cuda")
    for s in range(c["n_src"]):
        tr[s] = _arrivals((4, c["n_rcv"]), c["nt"], g)
    return {"traces": tr, "src": rs.randint(0, c["n_src"], c["events"]).astype(np.int32),
            "amps": np.exp(rs.standard_normal(c["events"])).astype(np.float32),
            "t0s": rs.uniform(0, c["span"], c["events"]).astype(np.float32), "dt": c["dt"],
            "n_out": c["nt"] + int(c["span"] / c["dt"])}


def _layout(c):
    F, H, K = (3 + 6 * c["nfreq"] + 7) // 8 * 8, c["hidden"], c["latent"]
    D = 4 * c["n_rcv"] * c["nt"]
    return F, H, K, D, [("W1", (F, H)), ("b1", (H,)), ("W2", (H, H)), ("b2", (H,)), ("W3", (H, K)), ("b3", (K,)),
                        ("Wd", (6 * K, D))]


_SCALE = (1.0e-1, 2.0e-8, 2.0e-8, 3.0e-8)  # pressure and velocities differ by orders of magnitude


def _network_inputs(c, seed):
    """A trained network's parameters (device, one vector), positions, moment tensors and, to train on, targets."""
    g = _gen(seed)
    F, H, K, D, segs = _layout(c)
    std = {"W1": 1 / math.sqrt(3 + 6 * c["nfreq"]), "W2": math.sqrt(2 / H), "W3": math.sqrt(1 / H),
           "Wd": 1 / math.sqrt(6 * K)}
    p = torch.zeros(sum(math.prod(s) for _, s in segs), device="cuda")
    o = 0
    for name, shape in segs:
        n = math.prod(shape)
        if name in std:
            for q in range(o, o + n, 1 << 28):  # in pieces: the decoder holds over a thousand million
                e = min(o + n, q + (1 << 28))
                p[q:e].normal_(0.0, std[name], generator=g)
        o += n
    n = c["batch"] * c.get("steps", 1)
    i = {"params": p, "pos": torch.rand((n, 3), device="cuda", generator=g) * 2 - 1,
         "mt": torch.randn((n, 6), device="cuda", generator=g)}
    i["mt"] /= (i["mt"][:, :3].square().sum(1) + 2 * i["mt"][:, 3:].square().sum(1)).sqrt()[:, None]
    if c["kind"] == "train":
        t = _arrivals((n, 4, c["n_rcv"]), c["nt"], g)
        i["target"] = t.mul_(torch.tensor(_SCALE, device="cuda")[None, :, None, None]).view(n, D)
    return i


_LR = 2.0e-6  # near the end of the cosine decay


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c}
    if kind == "run":
        i = _solver_inputs(c, seed, (c["nx"], c["ny"], c["nz"]), 1)
        s.update(model=_model(i), dt=i["dt"], pos=i["pos"][0], mt=i["mt"][0], w=i["w"])
        s["rcv"] = i["rcv"] if c["out"] == "host" else torch.from_numpy(i["rcv"]).cuda()
        s["traces"] = None if c["out"] == "host" else torch.empty((4, len(i["rcv"]), c["nt"]), device="cuda")
        s["fields"] = torch.empty((9,) + tuple(i["rho"].shape), device="cuda")
    elif kind == "catalog":
        i = _solver_inputs(c, seed, (c["n"],) * 3, c["nb"])
        # locations in sixes, each with the six unit moment tensors
        s.update(model=_model(i), dt=i["dt"], pos=np.repeat(i["pos"], 6, axis=0)[:c["nb"]],
                 mt=np.tile(np.eye(6), (c["nb"], 1))[:c["nb"]], w=np.tile(i["w"], (c["nb"], 1)),
                 rcv=torch.from_numpy(i["rcv"]).cuda(),
                 traces=torch.empty((c["nb"], 4, len(i["rcv"]), c["nt"]), device="cuda"))
    elif kind == "group":
        s.update(models=[], dts=[], srcs=[], rcvs=[], traces=[])
        for k, (n, nb) in enumerate(_sizes(c)):
            i = _solver_inputs(c, seed + 7 * k, (n,) * 3, nb)
            s["models"].append(_model(i))
            s["dts"].append(i["dt"])
            s["srcs"].append((i["pos"], i["mt"], np.tile(i["w"], (nb, 1))))
            s["rcvs"].append(torch.from_numpy(i["rcv"]).cuda())
            s["traces"].append(torch.empty((nb, 4, len(i["rcv"]), c["nt"]), device="cuda"))
    elif kind == "superpose":
        i = _superpose_inputs(c, seed)
        if c["entry"] == "host":
            i["traces"] = i["traces"].cpu().numpy()
            s["gather"] = None
        else:
            s["gather"] = torch.empty((4, c["n_rcv"], i["n_out"]), device="cuda")
        if c["entry"] == "noalloc":
            i.update({k: torch.from_numpy(i[k]).cuda() for k in ("src", "amps", "t0s")})
        s.update(i)
    elif kind in ("predict", "train"):
        i = _network_inputs(c, seed)
        net = surrogate.Surrogate(c["n_rcv"], c["nt"], nfreq=c["nfreq"], hidden=c["hidden"], latent=c["latent"],
                                  max_batch=c["batch"], seed=0)
        _set_params(net, i["params"])
        net.set_output_scale(_SCALE)
        s.update(net=net, pos=i["pos"], mt=i["mt"])
        if kind == "train":
            s.update(target=i["target"], params=i["params"])
        else:
            s["out"] = torch.empty((c["batch"], net.D), device="cuda")
    else:
        s["f"] = _velocity_model(c["nx"], c["ny"], c["nz"], c["dz"], seed)[0]
        s["out"] = torch.empty_like(s["f"])
    return s


def _set_params(net, p):
    rc = net.lib.es_sur_set_params(net._h, ctypes.c_void_p(p.data_ptr()))  # host or device memory
    if rc != 0:
        raise es.EsError(rc, "es_sur_set_params")


def _get_params(net, p):
    rc = net.lib.es_sur_get_params(net._h, ctypes.c_void_p(p.data_ptr()))
    if rc != 0:
        raise es.EsError(rc, "es_sur_get_params")
    return p


def run(state):
    s = state
    c, kind = s["case"], s["case"]["kind"]
    if kind == "run":
        m = s["model"]
        m.source_set(s["pos"], s["mt"], s["w"])
        m.state_reset()
        traces = m.run(c["nt"], s["dt"], s["rcv"], s["traces"])
        return {"traces": traces, "fields": m.state_get(s["fields"])}
    if kind == "catalog":
        s["model"].batch_set(s["pos"], s["mt"], s["w"])
        return {"traces": s["model"].run(c["nt"], s["dt"], s["rcv"], s["traces"])}
    if kind == "group":
        for m, (pos, mt, w) in zip(s["models"], s["srcs"]):
            m.batch_set(pos, mt, w)
        return {"traces": es.es_run_group(s["models"], c["nt"], s["dts"], s["rcvs"], s["traces"])}
    if kind == "superpose":
        if c["entry"] == "noalloc":
            return es.es_superpose_noalloc(s["traces"], s["src"], s["amps"], s["t0s"], s["dt"], s["n_out"], s["gather"])
        return es.es_superpose(s["traces"], s["src"], s["amps"], s["t0s"], s["dt"], s["n_out"], s["gather"])
    if kind == "predict":
        return s["net"].predict(s["pos"], s["mt"], s["out"])
    if kind == "train":
        b = c["batch"]
        for k in range(c["steps"]):
            q = slice(k * b, (k + 1) * b)
            s["net"].train_step(s["pos"][q], s["mt"][q], s["target"][q], _LR, want_loss=False)
        return _get_params(s["net"], s["params"])
    return es.es_laplacian(s["f"], (c["dx"], c["dy"], c["dz"]), s["out"])


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

def work(case):
    c, kind = case, case["kind"]
    if kind in ("run", "catalog", "group"):
        if kind == "run":
            grids = [((c["nx"], c["ny"], c["nz"]), 1)]
        else:
            grids = [((n,) * 3, nb) for n, nb in (_sizes(c) if kind == "group" else [(c["n"], c["nb"])])]
        b = f = 0.0
        for n, nb in grids:
            cs = float(n[0]) * n[1] * n[2] * nb * c["nt"]
            # the fields do not stay on the chip between the halves of a step: the velocity half reads 6 stresses
            # and the density and updates 3 velocities (13 arrays), the stress half reads 3 velocities, lambda and
            # mu and updates 6 stresses (17); simulations of one model share its materials
            b += cs * 4 * (12 + 15 + 3.0 / nb)
            # 18 derivatives (6 per axis): a real FFT forward and back, the multiply; then the updates
            f += cs * (sum(6 * (5 * math.log2(k) + 3) for k in n) + 60)
            b += 8.0 * 4 * c["rx"] * c["ry"] * c["nt"] * nb  # traces: recorded, laid out
        return {"bytes": b, "flops": f}
    if kind == "superpose":
        rows, n_out = 4 * c["n_rcv"], c["nt"] + int(c["span"] / c["dt"])
        used = c["n_src"] * (1 - (1 - 1 / c["n_src"]) ** c["events"]) if c["n_src"] > 1 else 1
        return {"bytes": 4.0 * rows * (used * c["nt"] + n_out), "flops": 2.0 * rows * c["nt"] * c["events"]}
    if kind in ("predict", "train"):
        F, H, K, D, segs = _layout(c)
        B, P = c["batch"], float(sum(math.prod(s) for _, s in segs))
        mlp = 2.0 * B * (F * H + H * H + H * K)
        if kind == "predict":
            return {"bytes": 2 * P + 4.0 * B * D, "flops": mlp + 2.0 * B * 6 * K * D}
        # FP32 parameters and two moments read and written once a step, the targets read; three decoder products
        return {"bytes": c["steps"] * (24 * P + 4.0 * B * D) + 4 * P,
                "flops": c["steps"] * 3 * (mlp + 2.0 * B * 6 * K * D)}
    n = float(c["nx"]) * c["ny"] * c["nz"]
    return {"bytes": 8 * n, "flops": n * sum(10 * math.log2(k) + 8 for k in (c["nx"], c["ny"], c["nz"]))}


# ---------------------------------------------------------------------------
# 64 bits
# ---------------------------------------------------------------------------

def _deriv64(f, dim, d, shift, cache):
    n = f.shape[dim]
    key = (dim, shift)
    if key not in cache:
        kap = 2 * math.pi * torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64) / (n * d)
        h = 1j * kap * torch.exp(0.5j * shift * d * kap)
        cache[key] = h.view([-1 if k == dim % f.dim() else 1 for k in range(f.dim())])
    return torch.fft.irfft(torch.fft.rfft(f, dim=dim) * cache[key], n=n, dim=dim)


def _harmonic64(*m):
    inv = sum(1.0 / x.clamp(min=1e-300) for x in m)
    ok = torch.ones_like(m[0], dtype=torch.bool)
    for x in m:
        ok &= x != 0
    return torch.where(ok, 4.0 / inv, torch.zeros_like(inv))


def _simulate64(i, pos, mt):
    """Traces [nb][4][n_rcv][nt] and final fields [nb][9][nz][ny][nx]: the split-field scheme with every split
    kept in 64 bits, derivatives by torch.fft."""
    rho, cp, cs = (i[k].double() for k in ("rho", "cp", "cs"))
    nb, nt, dt, L, tau = len(pos), i["nt"], i["dt"], i["pml"], i["tau"]
    ax = (-1, -2, -3)  # x, y, z
    up = lambda t, *dims: t.roll([-1] * len(dims), dims) if dims else t
    mu = cs * cs * rho
    lam = cp * cp * rho - 2 * mu
    b = [2 / (rho + up(rho, a)) for a in ax]
    mue = {}
    for p, q, f in ((0, 1, SXY), (0, 2, SXZ), (1, 2, SYZ)):
        mue[f] = _harmonic64(mu, up(mu, ax[p]), up(mu, ax[q]), up(mu, ax[p], ax[q]))
    cref = float(cp.max())
    P = {}
    for a in range(3):
        n = rho.shape[ax[a]]
        for st in (0, 1):
            x = np.arange(n) + 0.5 * st
            xi = np.where(x < L, (L - x) / L, np.where(x > n - 1 - L, (x - (n - 1 - L)) / L, 0)).clip(max=1)
            f = torch.from_numpy(np.exp(-2.0 * (cref / i["d"][a]) * xi ** 4 * dt / 2)).cuda()
            P[a, st] = f.view([-1 if k == 2 - a else 1 for k in range(3)])
    half = {VX: (0,), VY: (1,), VZ: (2,), SXX: (), SYY: (), SZZ: (), SXY: (0, 1), SXZ: (0, 2), SYZ: (1, 2)}
    shape = (nb,) + tuple(rho.shape)
    split = {(f, a): torch.zeros(shape, device="cuda", dtype=torch.float64) for f in range(9) for a in range(3)
             if not (f, a) in ((SXY, 2), (SXZ, 1), (SYZ, 0))}
    total = lambda f: sum(split[f, a] for a in range(3) if (f, a) in split)
    cache = {}

    def update(f, a, inc):
        p = P[a, int(a in half[f])]
        s = split[f, a]
        s.mul_(p).add_(inc).mul_(p)

    srcs = [[SXX, SXY, SXZ], [SXY, SYY, SYZ], [SXZ, SYZ, SZZ]]
    traces = torch.zeros((nb, 4, len(i["rcv"]), nt), device="cuda", dtype=torch.float64)
    r = torch.from_numpy(i["rcv"]).cuda().long()
    at = lambda t: t[:, r[:, 2], r[:, 1], r[:, 0]]
    k = torch.arange(nb, device="cuda")
    sx = [torch.from_numpy(pos[:, a].astype(np.int64)).cuda() for a in range(3)]
    m = torch.from_numpy(mt).cuda().float().double()
    w = i["w"].astype(np.float64)
    for n in range(nt):
        vold = [total(VX + c) for c in range(3)] if tau else None
        for a in range(3):
            for c in range(3):
                D = _deriv64(total(srcs[a][c]), ax[a], i["d"][a], 1 if a == c else -1, cache)
                update(VX + c, a, D.mul_(b[c]).mul_(dt))
        v = [total(VX + c) for c in range(3)]
        g = v if not tau else [dt * x + tau * (x - y) for x, y in zip(v, vold)]
        scale = 1.0 if tau else dt
        for a in range(3):
            D = _deriv64(g[a], ax[a], i["d"][a], -1, cache).mul_(scale)
            for c in range(3):
                update(SXX + c, a, (lam + 2 * mu if a == c else lam) * D)
            for c in range(3):
                if c != a:
                    f = {(0, 1): SXY, (0, 2): SXZ, (1, 2): SYZ}[min(a, c), max(a, c)]
                    update(f, a, _deriv64(g[c], ax[a], i["d"][a], 1, cache).mul_(scale).mul_(mue[f]))
        del g
        for c in range(6):
            s = split[SXX + c, 0 if (SXX + c, 0) in split else 1]
            s[k, sx[2], sx[1], sx[0]] += m[:, c] * float(w[n])
        traces[:, 0, :, n] = -sum(at(split[SXX + c, a]) for c in range(3) for a in range(3)) / 3
        for c in range(3):
            traces[:, 1 + c, :, n] = at(v[c])
    return traces, [total(f) for f in range(9)]


def _network64(c, i):
    """The network's layers in 64 bits: a dict of its parameters (views of one vector)."""
    p, o, W = i["params"], 0, {}
    for name, shape in _layout(c)[4]:
        n = math.prod(shape)
        W[name] = p[o:o + n].double().view(shape)
        o += n
    return W


def _forward64(c, W, pos, mt):
    pos, mt = pos.double(), mt.double()
    X = [pos]
    for j in range(c["nfreq"]):
        t = (math.pi * 2.0 ** j) * pos
        X.append(torch.stack([t.sin(), t.cos()], 2).view(len(pos), 6))
    X = torch.cat(X, 1)
    X = torch.nn.functional.pad(X, (0, W["W1"].shape[0] - X.shape[1]))
    h1 = (X @ W["W1"] + W["b1"]).clamp(min=0)
    h2 = (h1 @ W["W2"] + W["b2"]).clamp(min=0)
    a = h2 @ W["W3"] + W["b3"]
    z = (mt[:, :, None] * a[:, None, :]).reshape(len(pos), -1)
    return X, h1, h2, z


def _train64(c, i):
    W, B, K = _network64(c, i), c["batch"], c["latent"]
    scale = torch.tensor(_SCALE, device="cuda").double().repeat_interleave(c["n_rcv"] * c["nt"])
    m = {k: torch.zeros_like(v) for k, v in W.items()}
    v = {k: torch.zeros_like(x) for k, x in W.items()}
    for t in range(c["steps"]):
        q = slice(t * B, (t + 1) * B)
        X, h1, h2, z = _forward64(c, W, i["pos"][q], i["mt"][q])
        tau = i["target"][q].double() / scale
        dU = (z @ W["Wd"]).sub_(tau)
        dU.mul_((2.0 / B) / (tau.square().sum(1) + 1e-30)[:, None])
        del tau
        dz = (dU @ W["Wd"].T).view(B, 6, K)
        g = {"Wd": z.T @ dU}
        del dU
        da = (i["mt"][q].double()[:, :, None] * dz).sum(1)
        g["W3"], g["b3"] = h2.T @ da, da.sum(0)
        d2 = (da @ W["W3"].T) * (h2 > 0)
        g["W2"], g["b2"] = h1.T @ d2, d2.sum(0)
        d1 = (d2 @ W["W2"].T) * (h1 > 0)
        g["W1"], g["b1"] = X.T @ d1, d1.sum(0)
        for k in W:
            m[k].mul_(0.9).add_(g[k], alpha=0.1)
            v[k].mul_(0.999).addcmul_(g[k], g[k], value=0.001)
            W[k] = W[k] - _LR * (m[k] / (1 - 0.9 ** (t + 1))) / ((v[k] / (1 - 0.999 ** (t + 1))).sqrt_().add_(1e-8))
            del g[k]
    return torch.cat([W[k].reshape(-1) for k, _ in _layout(c)[4]])


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "run":
        i = _solver_inputs(c, seed, (c["nx"], c["ny"], c["nz"]), 1)
        tr, fields = _simulate64(i, i["pos"], i["mt"])
        return {"traces": tr[0], "fields": torch.stack([f[0] for f in fields])}
    if kind == "catalog":
        i = _solver_inputs(c, seed, (c["n"],) * 3, c["nb"])
        return {"traces": _simulate64(i, np.repeat(i["pos"], 6, axis=0)[:c["nb"]],
                                      np.tile(np.eye(6), (c["nb"], 1))[:c["nb"]])[0]}
    if kind == "group":
        out = []
        for k, (n, nb) in enumerate(_sizes(c)):
            i = _solver_inputs(c, seed + 7 * k, (n,) * 3, nb)
            out.append(_simulate64(i, i["pos"], i["mt"])[0])
        return {"traces": out}
    if kind == "superpose":
        i = _superpose_inputs(c, seed)
        g = torch.zeros((4, c["n_rcv"], i["n_out"]), device="cuda", dtype=torch.float64)
        for s, a, t0 in zip(i["src"], i["amps"], i["t0s"]):
            k = math.floor(float(t0) / c["dt"] + 0.5)
            n = min(c["nt"], i["n_out"] - k)
            if n > 0:
                g[:, :, k:k + n] += float(a) * i["traces"][int(s), :, :, :n].double()
        return g
    if kind in ("predict", "train"):
        i = _network_inputs(c, seed)
        if kind == "train":
            return _train64(c, i)
        W = _network64(c, i)
        z = _forward64(c, W, i["pos"], i["mt"])[3]
        scale = torch.tensor(_SCALE, device="cuda").double().repeat_interleave(c["n_rcv"] * c["nt"])
        return (z @ W["Wd"]).mul_(scale)
    f = _velocity_model(c["nx"], c["ny"], c["nz"], c["dz"], seed)[0].double()
    k = [2 * math.pi * torch.fft.fftfreq(n, d, device="cuda", dtype=torch.float64)
         for n, d in ((c["nz"], c["dz"]), (c["ny"], c["dy"]))]
    k.append(2 * math.pi * torch.fft.rfftfreq(c["nx"], c["dx"], device="cuda", dtype=torch.float64))
    k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
    return torch.fft.irfftn(-k2 * torch.fft.rfftn(f), s=f.shape)

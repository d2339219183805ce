"""The work a user has this library do, as cases that can be prepared, run and timed.

Twelve listed cases cover the public entry points over their real range: windows of LB steps on the
solver objects (single and half precision, both drives, both diffusion lattices), whole solves, batches,
the host-buffer solves, the setup of a structure (reconstruction, labelling, pore sizes, node set) and the
learned warm start (prediction and training step).  Sizes are those of synthetic.py's workloads and of the
benchmark's modes, with odd and ragged boxes among them; `draw` gives more cases of the same ranges.

Structures of the LB cases are packings of overlapping spheres made here from the seed, so that `exact` can
rebuild the same inputs and carry the method out in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

import paper_1410_1921_gb300 as P

WINDOW = 100  # LB steps per convergence check, the default of the solver parameters
F32, F16 = P.OM_F32, P.OM_F16DEV
SMALL_NET, WIDE_NET = "16,32,64,128", "32,64,128"  # the warm start's network; the network benchmark's


def _lb(kind, nx, ny, nz, porosity, mean, dx, **kw):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "porosity": porosity, "mean": mean, "dx": dx}
    c.update(kw)
    return c


def listed():
    def named(name, c):
        return dict(c, name=name)

    return [
        # the smallest workload (48^3 at 2 nm): a window of each model on solvers already made; launches count
        named("window_48", _lb("window", 48, 48, 48, 0.40, 20.0, 2.0, precision=F32, pressure=False, lattice=7)),
        # one structure solved with its check every 100 steps, an odd box of the size training structures have
        named("solve_61x67x75", _lb("solve", 61, 67, 75, 0.38, 22.0, 1.5, steps=1000)),
        # the porosity sweep's structure: the throughput workload, single precision
        named("window_256", _lb("window", 256, 256, 256, 0.35, 30.0, 1.0, precision=F32, pressure=False, lattice=7)),
        # the paper's own models at its own size: pressure ends and D3Q19 diffusion at 200^3, 1.5 nm
        named("paper_200", _lb("window", 200, 200, 200, 0.35, 45.0, 1.5, precision=F32, pressure=True, lattice=19)),
        # the large workload in half-precision storage
        named("half_512", _lb("window", 512, 512, 512, 0.30, 40.0, 1.0, precision=F16, pressure=False, lattice=7)),
        # training structures solved together: twenty boxes of mixed, ragged sizes
        named("batch_20", {"kind": "batch", "n": 20, "lo": 56, "hi": 80, "porosity": 0.36, "mean": 22.0, "dx": 1.5}),
        # both host-buffer solves, one window each, everything from labelling on inside the call
        named("host_256", _lb("host", 256, 256, 256, 0.35, 30.0, 1.0, steps=WINDOW)),
        # placing pore spheres until the porosity is reached
        named("reconstruct_256", _lb("reconstruct", 256, 256, 256, 0.35, 30.0, 1.0)),
        # a structure made ready for its solves: transport pores, chord pore sizes, node set
        named("pores_256", _lb("pores", 256, 256, 256, 0.35, 30.0, 1.0)),
        # the small workload's pore size (largest inscribed sphere), at twice its edge
        named("inscribed_96", _lb("inscribed", 96, 96, 96, 0.40, 20.0, 2.0)),
        # the trained network's prediction for one structure of an evaluation size, a ragged box
        named("predict_128", {"kind": "predict", "batch": 1, "nx": 128, "ny": 120, "nz": 136, "net": SMALL_NET, "out": 2}),
        # a training step's gradients on a batch of four
        named("train_4x64", {"kind": "train", "batch": 4, "nx": 64, "ny": 64, "nz": 64, "net": WIDE_NET, "out": 1}),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["window", "window", "window", "solve", "batch", "host", "reconstruct", "pores", "inscribed",
                       "predict", "train"])

    def box(lo, hi):
        e = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return [max(lo, min(hi, int(round(e * rng.uniform(0.8, 1.25))))) for _ in range(3)]

    por, dx = round(rng.uniform(0.28, 0.50), 3), rng.choice([1.0, 1.5])
    mean = round(rng.uniform(20.0, 45.0), 1)
    if kind == "window":
        paper = rng.random() < 0.3
        prec = F16 if not paper and rng.random() < 0.3 else F32
        return _lb("window", *box(40, 200 if paper else 300), por, mean, dx, precision=prec, pressure=paper,
                   lattice=19 if paper else 7)
    if kind == "solve":
        return _lb("solve", *box(32, 96), por, mean, dx, steps=100 * rng.randint(4, 12))
    if kind == "batch":
        lo = rng.randint(32, 64)
        return {"kind": "batch", "n": rng.randint(3, 24), "lo": lo, "hi": lo + rng.randint(4, 32), "porosity": por,
                "mean": mean, "dx": dx}
    if kind == "host":
        return _lb("host", *box(48, 256), por, mean, dx, steps=WINDOW)
    if kind in ("reconstruct", "pores"):
        return _lb(kind, *box(48, 288), round(rng.uniform(0.15, 0.45), 3), mean, dx)
    if kind == "inscribed":
        return _lb("inscribed", *box(32, 112), por, round(rng.uniform(15.0, 30.0), 1), 2.0)
    if kind == "predict":
        m = [8 * rng.randint(4, 20) for _ in range(3)]
        return {"kind": "predict", "batch": 1, "nx": m[0], "ny": m[1], "nz": m[2],
                "net": rng.choice([SMALL_NET, WIDE_NET]), "out": rng.choice([1, 2])}
    m = [8 * rng.randint(3, 10) for _ in range(3)]
    return {"kind": "train", "batch": rng.randint(1, 4), "nx": m[0], "ny": m[1], "nz": m[2],
            "net": rng.choice([SMALL_NET, WIDE_NET]), "out": rng.choice([1, 2])}


# ------------------------------------------------------------------ inputs, from the seed alone
def _balls(shape, mean, sd, porosity, rng):
    """Centres and radii (voxels) of overlapping spheres: no centre inside another sphere, y and z periodic,
    about half of them touching one already placed; enough for the porosity with overlaps to spare."""
    n = np.array(shape, float)
    centres, radii, vol = np.zeros((0, 3)), np.zeros(0), 0.0
    target = -math.log(1.0 - porosity) * float(np.prod(n)) * 1.3
    for _ in range(4000):
        k = 256
        c = rng.random((k, 3)) * n
        r = 0.5 * np.clip(rng.normal(mean, sd, k), mean - 3 * sd, mean + 3 * sd)
        must = rng.random(k) < 0.5
        if len(radii):
            d = c[:, None, :] - centres[None]
            d[..., 1:] -= n[1:] * np.round(d[..., 1:] / n[1:])
            dist = np.sqrt((d * d).sum(-1))
            ok = (dist >= np.maximum(r[:, None], radii[None])).all(1)
            ok &= ~must | (dist < r[:, None] + radii[None]).any(1)
        else:
            ok = np.ones(k, bool)
        new = []
        for i in np.flatnonzero(ok):
            if new:
                e = c[i] - c[new]
                e[:, 1:] -= n[1:] * np.round(e[:, 1:] / n[1:])
                if (np.sqrt((e * e).sum(-1)) < np.maximum(r[i], r[new])).any():
                    continue
            new.append(i)
        centres, radii = np.concatenate([centres, c[new]]), np.concatenate([radii, r[new]])
        vol += float((4.0 / 3.0 * math.pi * r[new] ** 3).sum())
        if vol >= target:
            break
    return centres, radii


def _pores(shape, mean, sd, porosity, seed):
    """uint8 pore mask on the GPU: the spheres in order until the porosity is reached, and one narrow channel
    along x so that something always spans the box."""
    rng = np.random.default_rng([seed, *shape])
    nx, ny, nz = shape
    centres, radii = _balls(shape, mean, sd, porosity, rng)
    m = torch.zeros(shape, dtype=torch.bool, device="cuda")
    y0, z0 = int(rng.integers(0, ny - 2)), int(rng.integers(0, nz - 2))
    m[:, y0:y0 + 2, z0:z0 + 2] = True
    every = max(1, len(radii) // 24)
    for i, (c, r) in enumerate(zip(centres, radii)):
        lo, hi = np.floor(c - r).astype(int), np.ceil(c + r).astype(int) + 1
        xs = torch.arange(max(0, lo[0]), min(nx, hi[0]), device="cuda")
        ys, zs = (torch.arange(lo[a], min(hi[a], lo[a] + shape[a]), device="cuda") for a in (1, 2))
        ball = ((xs + 0.5 - c[0]) ** 2)[:, None, None] + ((ys + 0.5 - c[1]) ** 2)[None, :, None] + \
            ((zs + 0.5 - c[2]) ** 2)[None, None, :] <= r * r
        at = (xs[:, None, None], (ys % ny)[None, :, None], (zs % nz)[None, None, :])
        m[at] = m[at] | ball
        if i % every == every - 1 and float(m.float().mean()) >= porosity:
            break
    return m.to(torch.uint8).contiguous()


def _structure(case, seed):
    mean = case["mean"] / case["dx"]
    shape = (case["nx"], case["ny"], case["nz"])
    return _pores(shape, max(5.0, min(mean, 0.6 * min(shape))), 0.25 * max(5.0, min(mean, 0.6 * min(shape))),
                  case["porosity"], seed)


def _fields(shape, seed):
    """A warm start's fields: a small velocity along x and a concentration near the linear profile."""
    nx, ny, nz = shape
    g = np.random.default_rng([seed, 77])
    a, b, c = g.random(3) * 2 * math.pi
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[:, None, None] / nx
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[None, :, None] / ny
    z = torch.arange(nz, device="cuda", dtype=torch.float64)[None, None, :] / nz
    wave = torch.sin(2 * math.pi * y + a) * torch.cos(4 * math.pi * z + b) + torch.sin(2 * math.pi * x + c)
    u = (1e-4 * (1.0 + 0.4 * wave)).float().reshape(-1).contiguous()
    conc = (1.0 - x + 0.1 * wave * x * (1.0 - x)).clamp(0.0, 1.0).float().expand(shape).reshape(-1).contiguous()
    return u, conc


def _shapes(case):
    """The batch's boxes."""
    g = np.random.default_rng([case["lo"], case["hi"], case["n"]])
    return [tuple(int(v) for v in g.integers(case["lo"], case["hi"] + 1, 3)) for _ in range(case["n"])]


def _flow_params(case, **kw):
    return P.flow_params(precision=case.get("precision", F32),
                         drive=P.OM_DRIVE_PRESSURE if case.get("pressure") else P.OM_DRIVE_FORCE, **kw)


def _diff_params(case, **kw):
    return P.diff_params(precision=case.get("precision", F32), lattice=case.get("lattice", 7), **kw)


def _recon_params(case):
    mean = case["mean"]
    return P.recon_params(mean, 0.25 * mean, 0.25 * mean, 1.75 * mean, case["porosity"], 0.3)


def _transport(mask, dom):
    tr = torch.empty(mask.numel(), dtype=torch.uint8, device="cuda")
    P.om_label_connectivity_dev(mask.reshape(-1), dom, None, tr)
    return tr


def _chords(mask, dom):
    d = torch.empty(mask.numel(), dtype=torch.float32, device="cuda")
    P.om_local_pore_diameter_dev(mask.reshape(-1), dom, P.OM_PORE_CHORD13, d)
    return d


def _net_inputs(case, seed):
    """Structures as the network sees them (mask and scaled pore size), targets and the loss mask."""
    shape = (case["nx"], case["ny"], case["nz"])
    xs, ts, ms = [], [], []
    for b in range(case["batch"]):
        m = _pores(shape, 14.0, 3.5, 0.35, seed + 1009 * b)
        u, c = _fields(shape, seed + 1009 * b)
        size = (0.2 + 0.3 * torch.sin(torch.arange(m.numel(), device="cuda") * 0.37).abs()).reshape(shape)
        xs.append(torch.stack([m.float(), m.float() * size], -1))
        ts.append(torch.stack([(u * 1e3).reshape(shape), c.reshape(shape)], -1)[..., :case["out"]])
        ms.append(m)
    return torch.stack(xs).contiguous(), torch.stack(ts).contiguous(), torch.stack(ms).contiguous()


def _convs(case):
    """Channels per level, and (stored inputs, outputs, inputs) of every 3x3x3 convolution in parameter order."""
    ch = [int(v) for v in case["net"].split(",")]
    convs = []
    for l, c in enumerate(ch):
        convs += [(16 if l == 0 else ch[l - 1], c, 2 if l == 0 else ch[l - 1]), (c, c, c)]
    for l in range(len(ch) - 2, -1, -1):
        convs += [(ch[l + 1] + ch[l], ch[l], ch[l + 1] + ch[l]), (ch[l], ch[l], ch[l])]
    return ch, convs


def _weights(case, seed):
    """The network's parameters: He-uniform convolutions, small biases and a head that is not zero."""
    ch, convs = _convs(case)
    g = torch.Generator().manual_seed(int(seed) + 12345)
    parts = []
    for cin, cout, fan in convs:
        parts.append((torch.rand(27 * cin * cout, generator=g) * 2 - 1) * math.sqrt(6.0 / (27 * fan)))
        parts.append(0.05 * torch.randn(cout, generator=g))
    parts.append(0.3 * torch.randn(ch[0] * case["out"], generator=g))
    parts.append(0.1 * torch.randn(case["out"], generator=g))
    return torch.cat(parts).cuda(), convs, ch


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    if kind in ("window", "solve"):
        shape = (case["nx"], case["ny"], case["nz"])
        mask, dom = _structure(case, seed), P.domain(shape, case["dx"])
        tr, d = _transport(mask, dom), _chords(mask, dom)
        s["ns"] = P.NodeSet(tr, dom)
        kw = {"conv_tol": 1e-12, "max_steps": case["steps"]} if kind == "solve" else {}
        s["flow"] = P.Flow(s["ns"], _flow_params(case, **kw))
        s["diff"] = P.Diffusion(s["ns"], d, _diff_params(case, **kw))
        s["u0"], s["c0"] = _fields(shape, seed)
        N = mask.numel()
        s["u"], s["c"], s["jx"] = (torch.empty(k * N, dtype=torch.float32, device="cuda") for k in (3, 1, 1))
    elif kind == "batch":
        doms, nodes, sizes, s["c0"], s["u0"], s["u"], s["c"] = [], [], [], [], [], [], []
        for k, shape in enumerate(_shapes(case)):
            mask = _structure(dict(case, nx=shape[0], ny=shape[1], nz=shape[2]), seed + 31 * k)
            dom = P.domain(shape, case["dx"])
            doms.append(dom)
            nodes.append(_transport(mask, dom))
            sizes.append(_chords(mask, dom))
            u, c = _fields(shape, seed + 31 * k)
            s["u0"].append(u)
            s["c0"].append(c)
            s["u"].append(torch.empty_like(u))
            s["c"].append(torch.empty_like(c))
        s["batch"] = P.Batch(doms, nodes, sizes, flow=_flow_params(case), diff=_diff_params(case))
    elif kind == "host":
        shape = (case["nx"], case["ny"], case["nz"])
        mask, s["dom"] = _structure(case, seed), P.domain(shape, case["dx"])
        s["mask"], s["d"] = mask.cpu().numpy(), _chords(mask, s["dom"]).cpu().numpy().reshape(shape)
        s["fp"], s["dp"] = (f(case, conv_tol=1e-12, max_steps=case["steps"]) for f in (_flow_params, _diff_params))
    elif kind == "reconstruct":
        s["dom"], s["seed"] = P.domain((case["nx"], case["ny"], case["nz"]), case["dx"]), int(seed)
        s["params"] = _recon_params(case)
        s["mask"] = torch.empty(case["nx"] * case["ny"] * case["nz"], dtype=torch.uint8, device="cuda")
    elif kind in ("pores", "inscribed"):
        s["dom"] = P.domain((case["nx"], case["ny"], case["nz"]), case["dx"])
        s["mask"] = _structure(case, seed).reshape(-1)
        s["tr"] = torch.empty_like(s["mask"])
        s["voxels"] = torch.zeros(s["mask"].numel(), dtype=torch.int64, device="cuda")  # as many as there are voxels
        s["d"] = torch.empty(s["mask"].numel(), dtype=torch.float32, device="cuda")
    else:
        x, t, m = _net_inputs(case, seed)
        w, _, ch = _weights(case, seed)
        s["net"] = P.UNet(2, case["out"], ch, seed=3)
        assert s["net"].n_params == w.numel()
        s["net"].set_params(w)
        s["x"], s["t"], s["m"] = x, t, m
        s["y"] = torch.empty(*x.shape[:4], case["out"], dtype=torch.float32, device="cuda")
        s["g"] = torch.empty_like(w)
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind == "window":  # a warm start, one check window of each model, and its fields
        s["flow"].init_velocity(s["u0"])
        s["flow"].step(WINDOW)
        s["flow"].get_velocity(s["u"])
        s["diff"].init_concentration(s["c0"])
        s["diff"].step(WINDOW)
        s["diff"].get_fields(s["c"], s["jx"])
        return {"u": s["u"], "c": s["c"], "jx": s["jx"]}
    if kind == "solve":  # a solve of each model from a warm start, to its step cap
        s["flow"].init_velocity(s["u0"])
        _, k, _ = s["flow"].solve()
        s["flow"].get_velocity(s["u"])
        s["diff"].init_concentration(s["c0"])
        _, D, _ = s["diff"].solve()
        s["diff"].get_fields(s["c"], s["jx"])
        return {"k": k, "u": s["u"], "D": D, "c": s["c"], "jx": s["jx"]}
    if kind == "batch":
        b = s["batch"]
        for model, start, out in ((0, s["u0"], s["u"]), (1, s["c0"], s["c"])):
            b.reset(model)
            for k, f in enumerate(start):
                b.init_fields(model, k, f)
            b.step(model, WINDOW)
            for k, f in enumerate(out):
                b.get_field(model, k, f)
        return {"u": s["u"], "c": s["c"]}
    if kind == "host":
        _, k, kl, _, _ = P.om_solve_permeability(s["mask"], s["dom"], s["fp"])
        _, D, tau, _, _ = P.om_solve_knudsen(s["mask"], s["d"], s["dom"], s["dp"])
        return {"k_lattice": kl, "D": D, "tau": tau}
    if kind == "reconstruct":
        st, eps, n = P.om_reconstruct_dev(s["seed"], s["dom"], s["params"], s["mask"])
        return {"mask": s["mask"], "porosity": eps, "spheres": n, "status": st}
    if kind == "pores":
        conn = P.om_label_connectivity_dev(s["mask"], s["dom"], None, s["tr"])
        P.om_local_pore_diameter_dev(s["mask"], s["dom"], P.OM_PORE_CHORD13, s["d"])
        ns = P.NodeSet(s["tr"], s["dom"])
        n = ns.n_nodes
        ns.voxels(s["voxels"])
        return {"transport": s["tr"], "connectivity": conn, "d": s["d"], "nodes": n, "voxels": s["voxels"]}
    if kind == "inscribed":
        P.om_local_pore_diameter_dev(s["mask"], s["dom"], P.OM_PORE_MIS, s["d"])
        return {"d": s["d"]}
    if kind == "predict":
        s["net"].forward(s["x"], s["y"])
        return {"y": s["y"]}
    loss = s["net"].backward(s["x"], s["t"], s["m"])
    s["net"].get_grads(s["g"])
    return {"loss": loss, "grads": s["g"]}


def _conv_flops(case):
    """Multiply-adds x 2 of one forward pass of the 3x3x3 convolutions."""
    ch = [int(v) for v in case["net"].split(",")]
    V, f = case["batch"] * case["nx"] * case["ny"] * case["nz"], 0
    for l, c in enumerate(ch):
        v = V // 8 ** l
        cin = 2 if l == 0 else ch[l - 1]
        f += v * 54 * (cin * c + c * c)
        if l + 1 < len(ch):
            f += v * 54 * ((ch[l + 1] + c) * c + c * c)
    return f


def work(case):
    """Bytes and operations of one pass.  An LB step takes the populations in and puts them out once (its input
    is the step before), so a window counts its steps; everything else counts its inputs and outputs once."""
    kind = case["kind"]
    if kind in ("predict", "train"):
        f = _conv_flops(case)
        V = case["batch"] * case["nx"] * case["ny"] * case["nz"]
        n = sum(27 * a * b + b for a, b, _ in _convs(case)[1])
        if kind == "predict":
            return {"bytes": 4 * V * (2 + case["out"]) + 4 * n, "flops": f}
        return {"bytes": 4 * V * (2 + case["out"]) + V + 8 * n, "flops": 3 * f}
    if kind == "batch":
        e = 0.5 * (case["lo"] + case["hi"])
        N = case["n"] * e ** 3
    else:
        N = case["nx"] * case["ny"] * case["nz"]
    if kind == "reconstruct":
        return {"bytes": N, "flops": 10 * N}
    nodes = 0.95 * case["porosity"] * N
    if kind == "pores":
        return {"bytes": N * (1 + 1 + 4) + 8 * nodes, "flops": 30 * N}
    if kind == "inscribed":
        return {"bytes": N * (1 + 4), "flops": 30 * N}
    b, q = (2 if case.get("precision", F32) == F16 else 4), case.get("lattice", 7)
    steps = case.get("steps", WINDOW)
    fields = 0 if kind == "host" else 4 * N * 7
    host = 6 * N if kind == "host" else 0
    return {"bytes": steps * nodes * (38 * b + 2 * q * b + 4) + fields + host, "flops": steps * nodes * (250 + 5 * q)}


# ------------------------------------------------------------------ exact: 64 bits, plain torch
_E19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, 1, 0), (1, -1, 0),
        (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1), (-1, 0, -1), (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1)]
_E7 = _E19[:7]


def _shift(a, e, fill):
    """b[v] = a[v + e]: y and z periodic, `fill` beyond the x faces."""
    b = torch.roll(a, (-e[1], -e[2]), (1, 2)) if e[1] or e[2] else a
    if e[0] == 0:
        return b
    out = torch.full_like(a, fill)
    if e[0] > 0:
        out[:-1] = b[1:]
    else:
        out[1:] = b[:-1]
    return out


def _spanning(mask):
    """Pores of the 18-connected components that reach both x faces (labels by hooking and pointer jumping)."""
    m = mask.bool()
    N = m.numel()
    lab = torch.full((N + 1,), N, dtype=torch.int32, device="cuda")
    lab[:N] = torch.where(m.view(-1), torch.arange(N, dtype=torch.int32, device="cuda"), N)
    while True:
        grid = lab[:N].view(m.shape)
        low = grid
        for e in _E19[1:]:
            low = torch.minimum(low, _shift(grid, e, N))
        new = lab.clone()
        new[:N] = torch.where(m, low, N).view(-1)
        new.scatter_reduce_(0, lab[:N].long(), new[:N].clone(), "amin")
        for _ in range(2):
            new = new[new.long()]
        if torch.equal(new, lab):
            break
        lab = new
    a, b = (torch.zeros(N + 1, dtype=torch.bool, device="cuda") for _ in range(2))
    a[lab[:N].view(m.shape)[0].reshape(-1).long()] = True
    b[lab[:N].view(m.shape)[-1].reshape(-1).long()] = True
    return (a & b)[lab[:N].long()].view(m.shape) & m


def _chord13(mask, dx):
    """Mean over the 13 lines of the all-pore length through each pore voxel, 64 bits."""
    m = mask.bool()
    nx, ny, nz = m.shape
    total = []
    for e in [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1),
              (1, 1, 1), (1, 1, -1), (1, -1, 1), (1, -1, -1)]:
        period = 0
        if e[0] == 0:
            period = ny if e[2] == 0 else nz if e[1] == 0 else ny * nz // math.gcd(ny, nz)
        limit = period or nx

        def runs(sign):
            r, k = m.int(), 1
            while k < limit:
                far, step = r, (sign * e[0] * k, sign * e[1] * k, sign * e[2] * k)
                far = torch.roll(far, (-step[1], -step[2]), (1, 2))
                if step[0]:
                    out = torch.zeros_like(far)
                    if abs(step[0]) < nx:
                        if step[0] > 0:
                            out[:-step[0]] = far[step[0]:]
                        else:
                            out[-step[0]:] = far[:step[0]]
                    far = out
                r, k = torch.where(r == k, r + far, r), 2 * k
            return r

        n = runs(1) + runs(-1) - 1
        if period:
            n = n.clamp(max=period)
        total.append(torch.where(m, n, 0).double())
    s = total[0] + total[1] + total[2] + math.sqrt(2.0) * sum(total[3:9]) + math.sqrt(3.0) * sum(total[9:])
    return s / 13.0 * dx


class _Lattice:
    """Gather tables of one set of boxes (nodes in voxel order, box after box) for a velocity set."""

    def __init__(self, boxes, E, periodic_x):
        self.E, self.opp = E, [E.index((-a, -b, -c)) for a, b, c in E]
        cols = [[] for _ in E]
        self.nf, at = sum(int(b.sum()) for b in boxes), 0
        self.x, self.nx = [], []
        for nodes in boxes:
            k = int(nodes.sum())
            idx = torch.full(nodes.shape, -1, dtype=torch.int32, device="cuda")
            idx[nodes] = torch.arange(at, at + k, dtype=torch.int32, device="cuda")
            own = idx[nodes]
            for i, e in enumerate(E):  # population i of a node comes from x - e_i, or bounces back
                if i == 0:
                    cols[0].append(own)
                    continue
                back = (-e[0], -e[1], -e[2])
                src = torch.roll(idx, (e[0], e[1], e[2]), (0, 1, 2)) if periodic_x else _shift(idx, back, -1)
                src = src[nodes]
                cols[i].append(torch.where(src >= 0, src + i * self.nf, own + self.opp[i] * self.nf))
                del src
            x = torch.arange(nodes.shape[0], device="cuda")[:, None, None].expand(nodes.shape)[nodes]
            self.x.append(x.int())
            self.nx.append(torch.full_like(self.x[-1], nodes.shape[0]))
            at += k
        self.src = [torch.cat(c) for c in cols]
        self.x, self.nx = torch.cat(self.x), torch.cat(self.nx)

    def stream(self, f, out):
        flat = f.view(-1)
        for i, s in enumerate(self.src):
            torch.index_select(flat, 0, s, out=out[i])


def _exact_flow(boxes, u0, tau, g, steps, drho=None):
    """u (3 x nodes) after `steps` D3Q19 steps from f_eq(1, (u0, 0, 0)), populations as deviations from w_i."""
    E, w = _E19, [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    lat = _Lattice(boxes, E, drho is None)
    nf, opp = lat.nf, lat.opp
    wp, wm = 1.0 / tau, 8.0 * (2.0 * tau - 1.0) / (8.0 * tau - 1.0)
    f = torch.empty(19, nf, dtype=torch.float64, device="cuda")
    for i, e in enumerate(E):
        f[i] = w[i] * (3.0 * e[0] * u0 + 4.5 * (e[0] * u0) ** 2 - 1.5 * u0 * u0)
    other = torch.empty_like(f)

    def moments(f):
        def along(a):
            p, q = [i for i, e in enumerate(E) if e[a] > 0], [i for i, e in enumerate(E) if e[a] < 0]
            s = f[p[0]] - f[q[0]]
            for i, j in zip(p[1:], q[1:]):
                s += f[i]
                s -= f[j]
            return s
        return f.sum(0), [along(0), along(1), along(2)]

    def feq(i, rho, u, sq):
        eu = sum(c * v for c, v in zip(E[i], u) if c)
        return w[i] * (rho + (3.0 * eu + 4.5 * eu * eu if i else 0.0) - 1.5 * sq)

    ends = []
    if drho is not None:  # Sec. 3.3: non-equilibrium extrapolation on the node layers x = 0 and x = nx - 1
        nodes = boxes[0]
        idx = torch.full(nodes.shape, -1, dtype=torch.int64, device="cuda")
        idx[nodes] = torch.arange(nf, device="cuda")
        for b, b1, b2, rho in ((idx[0], idx[1], idx[2], 0.5 * drho), (idx[-1], idx[-2], idx[-3], -0.5 * drho)):
            here = b >= 0
            ends.append((b[here], b1[here], b2[here], rho))

    def pressure(f):
        for b, b1, b2, rho in ends:
            has1, has2 = b1 >= 0, (b2 >= 0) & (b1 >= 0)
            f1, f2 = f[:, b1.clamp(min=0)], f[:, b2.clamp(min=0)]
            r1, j1 = moments(f1)
            _, j2 = moments(f2)
            ub = [torch.where(has2, 2 * p - q, p) * has1 for p, q in zip(j1, j2)]
            sqb, sq1 = sum(v * v for v in ub), sum(v * v for v in j1)
            for i in range(19):
                f[i, b] = feq(i, rho, ub, sqb) + torch.where(has1, f1[i] - feq(i, r1, j1, sq1), 0.0)

    for _ in range(steps):
        if ends:
            pressure(f)
        rho, u = moments(f)
        u[0] += 0.5 * g
        base = rho - 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        f[0] -= wp * (f[0] - w[0] * base)
        for i in range(1, 19):
            o = opp[i]
            if o < i:
                continue
            e = E[i]
            eu = sum((v if c > 0 else -v) for c, v in zip(e, u) if c)
            A = (0.5 * wp) * (f[i] + f[o]) - (wp * w[i]) * (base + 4.5 * eu * eu)
            B = (0.5 * wm) * (f[i] - f[o]) - (3.0 * w[i] * wm) * eu
            if e[0]:
                B -= w[i] * e[0] * (1.0 - 0.5 * wm) * 3.0 * g
            f[i] -= A + B
            f[o] -= A - B
        lat.stream(f, other)
        f, other = other, f
    _, u = moments(f)
    u[0] += 0.5 * g
    return torch.stack(u)


def _exact_diff(boxes, c0, omega, q, steps):
    """C and J_x (nodes) after `steps` steps from g = a C0 between the concentrations 1 and 0."""
    E = _E7 if q == 7 else _E19
    a = [1 / 4] + [1 / 8] * 6 if q == 7 else [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    lat = _Lattice(boxes, E, False)
    g = torch.stack([v * c0 for v in a])
    other = torch.empty_like(g)
    inlet, outlet = (lat.x == 0).nonzero().view(-1), (lat.x == lat.nx - 1).nonzero().view(-1)
    for _ in range(steps):
        c = g.sum(0)
        for i, v in enumerate(a):
            g[i] -= omega * (g[i] - v * c)
        lat.stream(g, other)
        for i, e in enumerate(E):
            if e[0] > 0:
                other[i, inlet] = -g[lat.opp[i], inlet] + 2.0 * a[i]
            elif e[0] < 0:
                other[i, outlet] = -g[lat.opp[i], outlet]
        g, other = other, g
    flux = sum(e[0] * g[i] for i, e in enumerate(E) if e[0])
    return g.sum(0), (1.0 - 0.5 * omega) * flux


def _spread(boxes, values):
    """Node values back on their voxels (0 elsewhere), one flat array per box."""
    out, at = [], 0
    for nodes in boxes:
        k = int(nodes.sum())
        v = torch.zeros(nodes.shape, dtype=torch.float64, device="cuda")
        v[nodes] = values[at:at + k]
        out.append(v.reshape(-1))
        at += k
    return out


def _omega(d):
    """Eq. 12 with d_ref = 60 nm and tau_ref = 1, pore sizes in single precision as the library takes them."""
    return 1.0 / (d.float().double() / 60.0 * 0.5 + 0.5)


def _to_si(D_lattice, T=300.0, M=0.016):
    """m^2/s of a D3Q7 diffusivity (Eqs. 11, 15)."""
    dk = 60e-9 / 3.0 * math.sqrt(8.0 * 8.314462618 * T / (math.pi * M))
    return D_lattice * dk / (0.25 * 0.5)


def _exact_net(case, seed):
    x, t, m = _net_inputs(case, seed)
    w, convs, ch = _weights(case, seed)
    w = w.double().requires_grad_(case["kind"] == "train")
    L, parts, at = len(ch), [], 0
    for cin, cout, _ in convs:
        parts.append((w[at:at + 27 * cin * cout].view(27, cin, cout), w[at + 27 * cin * cout:at + 27 * cin * cout + cout]))
        at += 27 * cin * cout + cout
    head, bias = w[at:at + ch[0] * case["out"]].view(ch[0], case["out"]), w[at + ch[0] * case["out"]:]

    def conv(v, k):  # v: [B, D, H, W, c]
        W, b = parts[k]
        p = torch.nn.functional.pad(v, (0, 0, 1, 1, 1, 1, 1, 1))
        D, H, Wd = v.shape[1:4]
        out = b.expand(*v.shape[:4], -1)
        for o in range(27):
            z, y, xx = o // 9, o // 3 % 3, o % 3
            out = out + p[:, z:z + D, y:y + H, xx:xx + Wd] @ W[o][:v.shape[-1]]
        return torch.relu(out)

    v, skips = x.double(), []
    for l in range(L):
        if l:
            B, D, H, Wd, c = v.shape
            v = v.view(B, D // 2, 2, H // 2, 2, Wd // 2, 2, c).mean((2, 4, 6))
        v = conv(conv(v, 2 * l), 2 * l + 1)
        skips.append(v)
    k = 2 * L
    for l in range(L - 2, -1, -1):
        up = v.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)
        v = conv(conv(torch.cat([up, skips[l]], -1), k), k + 1)
        k += 2
    y = v @ head + bias
    if case["kind"] == "predict":
        return {"y": y}
    keep = (m != 0)[..., None].double()
    loss = (keep * (y - t.double()) ** 2).sum() / (keep.sum() * case["out"])
    loss.backward()
    return {"loss": float(loss.detach()), "grads": w.grad}


def exact(case, seed):
    kind = case["kind"]
    if kind == "reconstruct":
        return None
    if kind in ("predict", "train"):
        return _exact_net(case, seed)
    if kind == "batch":
        shapes = _shapes(case)
        masks = [_structure(dict(case, nx=s[0], ny=s[1], nz=s[2]), seed + 31 * k) for k, s in enumerate(shapes)]
        start = [_fields(s, seed + 31 * k) for k, s in enumerate(shapes)]
    else:
        shapes = [(case["nx"], case["ny"], case["nz"])]
        masks = [_structure(case, seed)]
        start = [_fields(shapes[0], seed)]
    if kind == "inscribed":
        return {"d": _exact_inscribed(masks[0], case["dx"])}
    boxes = [_spanning(m) for m in masks]
    if kind == "pores":
        return {"transport": None, "connectivity": float(boxes[0].sum()) / float(masks[0].sum()),
                "d": _chord13(masks[0], case["dx"]).reshape(-1), "nodes": None, "voxels": None}
    sizes = torch.cat([_chord13(m, case["dx"])[b] for m, b in zip(masks, boxes)])
    omega = _omega(sizes)
    steps = case.get("steps", WINDOW)
    if kind == "host":
        x = torch.cat([torch.arange(s[0], device="cuda")[:, None, None].expand(s)[b] for s, b in zip(shapes, boxes)])
        u0, c0 = torch.zeros(x.numel(), dtype=torch.float64, device="cuda"), 1.0 - (x.double() + 0.5) / shapes[0][0]
    else:
        u0, c0 = (torch.cat([s[k].view(b.shape)[b].double() for s, b in zip(start, boxes)]) for k in (0, 1))
    drho = 1e-4 if case.get("pressure") else None
    u = _exact_flow(boxes, u0, 1.0, 0.0 if drho else 1e-6, steps, drho)
    c, j = _exact_diff(boxes, c0, omega, case.get("lattice", 7), steps)
    if kind == "batch":
        return {"u": _spread(boxes, u[0]), "c": _spread(boxes, c)}
    N, nx = masks[0].numel(), shapes[0][0]
    k, D = float(u[0].sum()) / N / 6.0 / 1e-6, float(j.sum()) / N * nx
    if kind == "host":
        mean = float((0.25 * (1.0 / omega - 0.5)).mean())
        return {"k_lattice": k, "D": _to_si(D), "tau": float(masks[0].sum()) / N * mean / D}
    fields = {"u": torch.cat([_spread(boxes, v)[0] for v in u]), "c": _spread(boxes, c)[0], "jx": _spread(boxes, j)[0]}
    return dict(fields, k=k, D=D) if kind == "solve" else fields


def _exact_inscribed(mask, dx):
    """Largest inscribed ball holding each pore voxel: d = dx (2 sqrt(r2) - 1)."""
    m = mask.bool()
    nx, ny, nz = m.shape
    far = 1 << 28
    r2 = torch.where(m, far, 0).int()
    for axis, n in ((2, nz), (1, ny)):
        best = r2.clone()
        for k in range(1, n // 2 + 1):
            for s in (k, -k):
                best = torch.minimum(best, torch.roll(r2, s, axis) + k * k)
        r2 = best
    best = r2.clone()
    for k in range(1, nx):
        best[k:] = torch.minimum(best[k:], r2[:-k] + k * k)
        best[:-k] = torch.minimum(best[:-k], r2[k:] + k * k)
    r2 = best
    top = int(r2.max())
    R = math.isqrt(max(0, top - 1))
    out = torch.zeros_like(r2)
    for a in range(-min(R, nx - 1), min(R, nx - 1) + 1):
        for b in range(-min(R, ny // 2), min(R, ny // 2) + 1):
            for c in range(-min(R, nz // 2), min(R, nz // 2) + 1):
                k = a * a + b * b + c * c
                if k >= top:
                    continue
                moved = torch.roll(r2, (b, c), (1, 2)) if b or c else r2
                if a > 0:
                    moved, here = moved[:-a], out[a:]
                elif a < 0:
                    moved, here = moved[-a:], out[:a]
                else:
                    here = out
                here.copy_(torch.maximum(here, torch.where(moved > k, moved, 0)))
    return torch.where(m, (2.0 * out.double().sqrt() - 1.0) * dx, 0.0).reshape(-1)

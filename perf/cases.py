"""Workloads of the RD-CNN framework for performance measurement.

Each case is one call sequence of a user's program through the public API, over
the range of sizes, plane types, boundaries, cell models and directions that
the library is used for:

* ``run``        load a state, apply Eq. 1 T times, read the state (Grid.run);
* ``snapshots``  the same with the state captured every few steps (the paper's main loop);
* ``sweep``      a parameter search: a batch of instances of several sizes, each
                 with its own gene, advanced together and ranked by statistics (Batch);
* ``train``      forward and backward of a loss on the final state (RDCNNFunction).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2102_10340_gb300 as rd

DEV = "cuda"
DTYPES = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16, "f16": torch.float16}
GENE = {"dt": 0.1, "a": -0.3, "b": 1.3, "eps": -0.1, "c": 1.0, "Du": 0.06, "Dv": 1.0}
# Chua-Yang cell: feedback centre 2, arms 0.25 (a smoothing / edge-keeping template)
CENN = {"dt": 0.1, "a": 0.0, "b": 0.0, "eps": 0.0, "c": 2.0, "Du": 0.25, "Dv": 0.0}
SIDES = (128, 256, 512, 1024)  # instance sides of a sweep


def _run(name, nn, nm, T, dtype="f32", variant="auto", reaction="fhn", boundary="periodic", init="uniform"):
    return {"name": name, "kind": "run", "nn": nn, "nm": nm, "T": T, "dtype": dtype, "variant": variant,
            "reaction": reaction, "boundary": boundary, "init": init}


def listed():
    return [
        # the paper's small array, all cells random: a run is many short launches
        _run("small_64", 64, 64, 1000),
        # one point of an interactive search at the search harness' size
        _run("search_256", 256, 256, 1000, init="patch"),
        # image processing on a 1024 x 1024 picture (edge detection to steady state)
        _run("image_1024", 1024, 1024, 1000, init="smooth"),
        # slow growth from a random square in the middle of a large array: the headline workload
        _run("growth_4096", 4096, 4096, 1000, init="patch"),
        # a picture whose sides are what the camera gave: odd, so rows are not vector-aligned
        _run("ragged_1003x1021", 1003, 1021, 100),
        # cellular neural network on a picture without wrap-around
        _run("cenn_zeroflux_2048", 2048, 2048, 200, reaction="cenn", boundary="zeroflux", init="smooth"),
        # half the memory per cell and the paper's one step per launch (one rounding a step)
        _run("step_bf16_4096", 4096, 4096, 50, dtype="bf16", variant="step1"),
        # double precision reference runs
        _run("reference_f64_512", 512, 512, 200, dtype="f64"),
        # frames for a film, one every 20 steps, kept on the device
        {"name": "film_1024x768", "kind": "snapshots", "nn": 768, "nm": 1024, "T": 200, "every": 20, "dtype": "f32",
         "reaction": "fhn", "boundary": "zeroflux", "init": "patch"},
        # a (Du, Dv) x gene search over arrays of four sizes, ranked on the device
        {"name": "sweep_24", "kind": "sweep", "n": 24, "T": 80, "sizes": 4, "dtype": "f32", "boundary": "periodic"},
        # fitting the gene and the initial state to a target picture, single precision
        {"name": "train_512", "kind": "train", "nn": 512, "nm": 512, "T": 60, "dtype": "f32", "boundary": "periodic"},
        # the same in double precision, without wrap-around, on a small array
        {"name": "train_f64_128", "kind": "train", "nn": 128, "nm": 128, "T": 100, "dtype": "f64", "boundary": "zeroflux"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi, unit):
    return max(unit, _log(rng, lo, hi) // unit * unit)


def draw(rng):
    kind = rng.choice(["run"] * 6 + ["snapshots", "sweep", "train", "train"])
    boundary = rng.choice(["periodic", "periodic", "zeroflux"])
    if kind == "sweep":
        return {"kind": kind, "n": rng.randint(3, 24), "T": _log(rng, 20, 80), "sizes": rng.randint(1, 4),
                "dtype": "f32", "boundary": boundary}
    if kind == "train":
        dtype = rng.choice(["f32", "f32", "f64"])
        unit = 4 if dtype == "f32" else 2
        nn, nm = _side(rng, 48, 512, 1), _side(rng, 48, 512, unit)
        most = 5e7 if dtype == "f32" else 1.6e6  # cell-steps
        return {"kind": kind, "nn": nn, "nm": nm, "T": max(4, min(_log(rng, 20, 60), int(most / (nn * nm)))),
                "dtype": dtype, "boundary": boundary}
    if kind == "snapshots":
        nn, nm = _side(rng, 64, 1024, rng.choice([1, 16])), _side(rng, 64, 1024, rng.choice([1, 4, 32]))
        T = _log(rng, 40, 100)
        return {"kind": kind, "nn": nn, "nm": nm, "T": T, "every": rng.randint(max(2, T // 12), T), "dtype": "f32",
                "reaction": "fhn", "boundary": boundary, "init": rng.choice(["patch", "uniform"])}
    dtype, variant = rng.choice([("f32", "auto")] * 6 + [("f64", "auto"), ("bf16", "step1"), ("f16", "step1"),
                                                         ("f32", "step1")])
    aligned = variant == "step1" or rng.random() < 0.6
    nn, nm = _side(rng, 48, 4096, rng.choice([1, 16])), _side(rng, 48, 4096, rng.choice([8, 32]) if aligned else 1)
    most = 4e9 if aligned else 5e8  # cell-steps
    if dtype == "f64":
        most = 5e7
    elif variant == "step1":
        most = 8e8
    reaction = "cenn" if boundary == "zeroflux" and rng.random() < 0.5 else "fhn"
    init = rng.choice(["uniform", "smooth", "patch", "patch"])
    # Between about 120 and 600 steps the random starts of the FitzHugh-Nagumo cell pass their separatrix,
    # where a few cells magnify any rounding a thousandfold: those runs are compared before it.
    T = _log(rng, 20, 1000 if reaction == "cenn" or init == "patch" else 100)
    return {"kind": "run", "nn": nn, "nm": nm, "T": max(2, min(T, int(most / (nn * nm)))), "dtype": dtype,
            "variant": variant, "reaction": reaction, "boundary": boundary, "init": init}


# ---------------------------------------------------------------------- inputs

def _image(init, seed, nn, nm):
    """x in [-1, 1] as float64 on the device: all cells random, a random 16 x 16 square in the
    middle of zeros, or a blurred random picture (periodic Gaussian, 8 pixels)."""
    gen = torch.Generator(device=DEV).manual_seed(1000003 * (seed + 1) + 17)
    if init == "patch":
        x = torch.zeros((nn, nm), dtype=torch.float64, device=DEV)
        p = min(16, nn, nm)
        r, c = nn // 2 - p // 2, nm // 2 - p // 2
        x[r:r + p, c:c + p] = 2 * torch.rand((p, p), generator=gen, dtype=torch.float64, device=DEV) - 1
        return x
    x = torch.rand((nn, nm), generator=gen, dtype=torch.float64, device=DEV)
    if init == "smooth":
        ky = torch.fft.fftfreq(nn, dtype=torch.float64, device=DEV)[:, None]
        kx = torch.fft.fftfreq(nm, dtype=torch.float64, device=DEV)[None, :]
        x = torch.fft.ifft2(torch.fft.fft2(x) * torch.exp(-2.0 * (8 * math.pi) ** 2 * (kx * kx + ky * ky))).real
        x = (x - x.min()) / (x.max() - x.min())
    return 2 * x - 1


def _gene(case):
    return dict(CENN if case.get("reaction") == "cenn" else GENE)


def _instances(case, seed):
    """Sizes from the case, genes around the defaults from the seed (Sec. III.A's plane)."""
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["n"]):
        side = SIDES[(i * 7 + 3) % case["sizes"]]
        s = rng.uniform(0.8, 1.2, size=4)
        gene = dict(GENE, a=GENE["a"] * s[0], b=GENE["b"] * s[1], eps=GENE["eps"] * s[2], c=GENE["c"] * s[3],
                    Du=rng.uniform(0.01, 0.25), Dv=rng.uniform(0.01, 0.25))
        out.append({"nn": side, "nm": side, "params": gene})
    return out


def _start(case, seed):
    """The picture x in the case's plane type."""
    return _image(case.get("init", "uniform"), seed, case["nn"], case["nm"]).to(DTYPES[case["dtype"]])


def _target(case, seed):
    i = (torch.arange(case["nn"], device=DEV)[:, None] + seed % 32) // 16
    j = (torch.arange(case["nm"], device=DEV)[None, :] + seed % 29) // 16
    return torch.where((i + j) % 2 == 0, 1.0, -1.0).to(DTYPES[case["dtype"]])


def prepare(case, seed):
    kind, dtype = case["kind"], DTYPES[case["dtype"]]
    if kind == "sweep":
        specs = _instances(case, seed)
        batch = rd.Batch(specs, dtype=dtype, device=DEV, boundary=case["boundary"])
        starts = [_image("uniform", seed + 31 * i, s["nn"], s["nm"]).to(dtype) for i, s in enumerate(specs)]
        return {"case": case, "batch": batch, "starts": starts}
    if kind == "train":
        x = _start(case, seed)
        theta = torch.tensor([GENE[k] for k in rd.GRAD_NAMES], dtype=torch.float64)
        return {"case": case, "u0": x, "v0": 0.5 * x, "theta": theta, "target": _target(case, seed)}
    grid = rd.Grid(case["nn"], case["nm"], _gene(case), dtype=dtype, reaction=case["reaction"], device=DEV,
                   boundary=case["boundary"])
    state = {"case": case, "grid": grid, "x": _start(case, seed)}
    if kind == "snapshots":
        shape = (case["T"] // case["every"] + 1, case["nn"], case["nm"])
        state["frames"] = tuple(torch.empty(shape, dtype=dtype, device=DEV) for _ in range(2))
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "run":
        g = state["grid"]
        g.init(state["x"])
        g.run(case["T"], variant=case["variant"])
        return {"u": g.u, "v": g.v}
    if kind == "snapshots":
        g = state["grid"]
        g.init(state["x"])
        us, vs = g.run_snapshots(case["T"], case["every"], out="device", buffers=state["frames"])
        return {"u": us, "v": vs}
    if kind == "sweep":
        b = state["batch"]
        for i, x in enumerate(state["starts"]):
            b.set_state(i, x, x)
        b.run(case["T"])
        stats = b.summary()
        return {"states": [list(b.state(i)) for i in range(len(b))], "stats": stats}
    u0 = state["u0"].detach().requires_grad_(True)
    v0 = state["v0"].detach().requires_grad_(True)
    theta = state["theta"].detach().requires_grad_(True)
    uT, vT = rd.RDCNNFunction.apply(u0, v0, theta, case["T"], GENE["dt"], 0, case["boundary"])
    loss = ((uT - state["target"]) ** 2).mean()
    gu, gv, gt = torch.autograd.grad(loss, (u0, v0, theta))
    return {"u": uT.detach(), "v": vT.detach(), "du0": gu, "dv0": gv, "dtheta": gt}


# ---------------------------------------------------------------------- floors and tolerances

# Arithmetic of one cell-step: FitzHugh-Nagumo 2 x (3 add + 1 fma) + 7 + 4; Chua-Yang 4 outputs + sum + update.
_FLOPS = {"fhn": 27, "cenn": 17}


def work(case):
    esz = DTYPES[case["dtype"]].itemsize
    if case["kind"] == "sweep":
        cells = sum(s["nn"] * s["nm"] for s in _instances(case, 0))
        return {"bytes": 4 * cells * esz, "flops": 27 * cells * case["T"]}
    cells = case["nn"] * case["nm"]
    flops = _FLOPS[case.get("reaction", "fhn")] * cells * case["T"]
    if case["kind"] == "train":  # u0, v0, target in; uT, vT and two gradients out; the reverse step adds six sums
        return {"bytes": 7 * cells * esz, "flops": flops + 39 * cells * case["T"]}
    planes = 1 + 2 * (case["T"] // case["every"] + 1 if case["kind"] == "snapshots" else 1)
    if case.get("variant") == "step1":  # the caller asks for one pass over memory per step
        planes += 4 * (case["T"] - 1) + 2
    return {"bytes": planes * cells * esz, "flops": flops}


def tolerance(case):
    """About four times the largest error against exact() seen over the listed cases and 36 drawn
    ones: f64 5e-14 (normwise; single cells 3e-12), 16-bit planes 2.4e-4 (single cells 5e-2: a value
    next to a rounding boundary goes to its other neighbour), f32 2.5e-6 (single cells 1.8e-4)."""
    if case["dtype"] == "f64":
        return {"rel": 2e-13, "max": 1e-11}
    if case["dtype"] in ("bf16", "f16"):
        return {"rel": 1e-3, "max": 0.2}
    return {"rel": 1e-5, "max": 7e-4}


# ---------------------------------------------------------------------- the same results in 64 bits

def _shift(x, d, axis, boundary):
    if boundary == "periodic":
        return torch.roll(x, d, axis)
    n = x.shape[axis]
    edge = x.narrow(axis, 0, 1) if d > 0 else x.narrow(axis, n - 1, 1)
    rest = x.narrow(axis, 0, n - 1) if d > 0 else x.narrow(axis, 1, n - 1)
    return torch.cat([edge, rest] if d > 0 else [rest, edge], dim=axis)


def _nbrs(x, boundary):
    return (_shift(x, 1, 0, boundary) + _shift(x, -1, 0, boundary)) + (_shift(x, 1, 1, boundary) + _shift(x, -1, 1, boundary))


def _step(u, v, g, reaction, boundary):
    if reaction == "cenn":
        y = u.clamp(-1.0, 1.0)
        return u + g["dt"] * (-u + g["c"] * y + g["Du"] * _nbrs(y, boundary) + v), v
    fu = g["c"] * u - u * u * u / 3.0 - v
    fv = -g["eps"] * (u - g["b"] * v + g["a"])
    return (u + g["dt"] * (fu + g["Du"] * (_nbrs(u, boundary) - 4.0 * u)),
            v + g["dt"] * (fv + g["Dv"] * (_nbrs(v, boundary) - 4.0 * v)))


def _stats(u, v, threshold=0.05):
    grad = (torch.roll(u, -1, 0) - u).abs() + (torch.roll(u, -1, 1) - u).abs()
    return torch.stack([u.mean(), u.var(unbiased=False), u.min(), u.max(), v.mean(), v.var(unbiased=False), grad.mean(),
                        (grad > threshold).double().mean()])


def exact(case, seed):
    kind, boundary, T = case["kind"], case["boundary"], case["T"]
    if kind == "sweep":
        states, stats = [], []
        for i, s in enumerate(_instances(case, seed)):
            u = _image("uniform", seed + 31 * i, s["nn"], s["nm"]).to(DTYPES[case["dtype"]]).double()
            v = u.clone()
            for _ in range(T):
                u, v = _step(u, v, s["params"], "fhn", boundary)
            states.append([u, v])
            stats.append(_stats(u, v))
        return {"states": states, "stats": torch.stack(stats).cpu()}
    if kind == "train":
        x = _start(case, seed)
        u0 = x.double().clone().requires_grad_(True)
        v0 = (0.5 * x).double().clone().requires_grad_(True)
        theta = torch.tensor([GENE[k] for k in rd.GRAD_NAMES], dtype=torch.float64, device=DEV, requires_grad=True)
        g = dict(zip(rd.GRAD_NAMES, theta.unbind()), dt=GENE["dt"])
        u, v = u0, v0
        for _ in range(T):
            u, v = _step(u, v, g, "fhn", boundary)
        loss = ((u - _target(case, seed).double()) ** 2).mean()
        gu, gv, gt = torch.autograd.grad(loss, (u0, v0, theta))
        return {"u": u.detach(), "v": v.detach(), "du0": gu, "dv0": gv, "dtheta": gt.cpu()}
    g, reaction, dtype = _gene(case), case["reaction"], DTYPES[case["dtype"]]
    u = _start(case, seed).double()
    v = u.clone()
    us, vs = [u], [v]
    for t in range(1, T + 1):
        u, v = _step(u, v, g, reaction, boundary)
        if dtype.itemsize == 2:  # the state lives in 16-bit planes: rounded when a step stores it
            u, v = u.to(dtype).double(), v.to(dtype).double()
        if kind == "snapshots" and t % case["every"] == 0:
            us.append(u)
            vs.append(v)
    if kind == "snapshots":
        return {"u": torch.stack(us), "v": torch.stack(vs)}
    return {"u": u, "v": v}

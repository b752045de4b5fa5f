"""The work that a user of this framework has it do, as cases to be measured.

Every case goes through the public entry points (the binding in ``_lib``, the
autograd function, the CUDA graph of the batched push) at sizes of this
repository's own workloads, tests and benchmark: the six particle workloads of
``workloads.config`` with their ensembles and step counts scaled so that a pass
takes milliseconds, the grid-node evaluation and the Sec. 4 lines of the
benchmark, and the packing of a static grid.

``listed`` names the fixed cases, ``draw`` gives more of the same ranges,
``prepare`` makes a case's inputs on the GPU from a seed, ``run`` is one pass,
``work`` counts what a pass cannot do without, and ``exact`` computes the
outputs of a pass in 64 bits with plain torch.

An FP32 push accumulates float velocities into positions that are stored in
double, so its positions and the means of its gammas are good to float, and
``run`` hands them on in float, as a particle dump does.  The FP64 push returns
its state as it is.
"""
import math

import numpy as np
import torch

from paper_2307_04843_gb300 import _lib, autograd, workloads

L = workloads.LAMBDA
DT = workloads.DT


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: one step of a user's own time loop over a small ensemble
        # (launch and host path), the default launch shape
        dict(name="step_1k", op="push", workload=2, n=1000, steps=1, precision="fp32", grid=0, launch="default",
             t0=-6.0, loop=True),
        # workload 1 as it stands: 1e4 electrons, 2000 steps, plain FP64, light-front invariant per step
        dict(name="plane_fp64_10k", op="push", workload=1, n=10_000, steps=2000, precision="fp64", grid=0,
             launch="default", t0=0.0, lightfront=True),
        # the README's example: 1e6 electrons, Gaussian beam plus the 256^3 static grid, no launch shape set
        dict(name="gauss_grid_1m", op="push", workload=2, n=1_000_000, steps=400, precision="fp32", grid=256,
             launch="default", t0=-6.0),
        # workload 2, the benchmark's headline, with the launch shape the autotuner picks for it
        dict(name="gauss_grid_4m", op="push", workload=2, n=4_000_000, steps=400, precision="fp32", grid=256,
             launch="tuned", t0=-6.0),
        # workload 3: counter-propagating beam through a circularly polarised LG_{1,2} pulse
        dict(name="ics_lg_3m", op="push", workload=3, n=3_200_000, steps=300, precision="fp32", grid=0,
             launch="tuned", t0=27.0),
        # workload 4: flying focus of 64 spectral components
        dict(name="flying_1m", op="push", workload=4, n=1_000_000, steps=200, precision="fp32", grid=0,
             launch="tuned", t0=630.0),
        # workload 5: 256 Gaussian sets of uneven size in one persistent launch, replayed from a CUDA graph
        dict(name="batched_256", op="batch", n_sets=256, n=4_000_000, steps=500, launch="tuned", graph=True, t0=-5.0),
        # gradients of workload 5's mean final gamma (forward, checkpoints, reverse) through torch.autograd
        dict(name="adjoint_64", op="adjoint", n_sets=64, n=1_000_000, steps=200, ckpt=100, t0=-2.0),
        # E1/B1 on the staggered nodes of a 256^3 Yee grid (the grid-node form of the technique)
        dict(name="nodes_gauss_256", op="nodes", kind="gauss", nx=256, ny=256, nz=256, precision="fp32",
             dtype="float32", accumulate=False),
        # Sec. 4 lines of the benchmark: the split line, E1 and J1 evaluated in the kernel every step
        dict(name="split_line", op="line", form="split", n_lines=304, nz=4096, steps=500, dtype="float32"),
        # and the traditional Yee line with the plasma current that Sec. 4 compares it with
        dict(name="plasma_line", op="line", form="plasma", n_lines=304, nz=4096, steps=5000, dtype="float32"),
        # per-cell coefficient copy of a 256^3 grid, made anew whenever a user's grid field changes
        dict(name="pack_cells_256", op="pack", layout="cells", nx=256, ny=256, nz=256),
    ]


def _size(rng, lo, hi):
    """A size in [lo, hi], uniform in its logarithm; odd ones among them."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["push", "push", "push", "push", "batch", "sweep", "adjoint", "nodes", "line", "line", "pack"])
    if op == "push":
        w = rng.choice([1, 2, 2, 3, 4])
        precision = rng.choice({1: ["fp64", "fp32"], 2: ["fp32", "fp32", "fp32", "fp32_phase64", "fp64"],
                                3: ["fp32"], 4: ["fp32"]}[w])
        n = _size(rng, 200, {"fp64": 30_000, "fp32_phase64": 500_000,
                             "fp32": {1: 3_000_000, 2: 4_000_000, 3: 3_000_000, 4: 800_000}[w]}[precision])
        steps = _size(rng, 20, 200 if w == 4 else 300)
        grid = rng.choice([0, _size(rng, 24, 256)]) if w == 2 else 0
        return dict(op="push", workload=w, n=n, steps=steps, precision=precision, grid=grid,
                    launch=rng.choice(["default", "tuned"]) if precision == "fp32" else "default",
                    t0={1: 0.0, 2: -6.0, 3: 27.0, 4: 630.0}[w])
    if op == "batch":
        s = _size(rng, 3, 256)
        return dict(op="batch", n_sets=s, n=_size(rng, 40 * s, 4_000_000), steps=_size(rng, 20, 400),
                    launch=rng.choice(["default", "tuned"]), graph=rng.random() < 0.5, t0=-5.0)
    if op == "sweep":
        return dict(op="sweep", n=_size(rng, 3000, 3_000_000), steps=_size(rng, 20, 400),
                    launch=rng.choice(["default", "tuned"]), t0=-4.0)
    if op == "adjoint":
        s = _size(rng, 1, 128)
        return dict(op="adjoint", n_sets=s, n=_size(rng, max(500, 60 * s), 1_000_000), steps=_size(rng, 20, 200),
                    ckpt=_size(rng, 10, 100), t0=-2.0)
    if op == "nodes":
        return dict(op="nodes", kind=rng.choice(["gauss", "gauss", "plane", "lg"]), nx=_size(rng, 20, 256),
                    ny=_size(rng, 20, 256), nz=_size(rng, 20, 256), precision="fp32", dtype="float32",
                    accumulate=rng.random() < 0.3)
    if op == "line":
        form = rng.choice(["split", "plasma", "yee"])
        return dict(op="line", form=form, n_lines=_size(rng, 1, 304), nz=_size(rng, 300, 8192 if form == "yee" else 6144),
                    steps=_size(rng, 50, 300 if form == "split" else 3000), dtype="float32")
    return dict(op="pack", layout=rng.choice(["cells", "cells", "nodes"]), nx=_size(rng, 20, 256),
                ny=_size(rng, 20, 256), nz=_size(rng, 20, 256))


# --------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + 17)
    return g


def _uniform(n, box, g):
    lo = torch.tensor([b[0] for b in box], dtype=torch.float64, device="cuda")[:, None]
    hi = torch.tensor([b[1] for b in box], dtype=torch.float64, device="cuda")[:, None]
    r = torch.rand((3, n), dtype=torch.float64, device="cuda", generator=g)
    return [v.clone() for v in lo + r * (hi - lo)]  # each array in an allocation of its own


def _ensemble(case, seed):
    """Initial particles (x, y, z double; u in the arithmetic of the push)."""
    g, n = _gen(seed), case["n"]
    udt = torch.float64 if case.get("precision", "fp32") == "fp64" else torch.float32
    if case["op"] == "push" and case["workload"] == 3:
        # gamma ~ N(1000, 10), 1 mrad, moving along -z; the centre crosses the focus at t = 30
        b = workloads.config(3)["beam"]
        r = torch.randn((6, n), dtype=torch.float64, device="cuda", generator=g)
        x, y = b["sigma_perp"] * r[0], b["sigma_perp"] * r[1]
        z = (30.0 - case["t0"]) + b["sigma_z"] * r[2]
        gam = b["gamma_mean"] + b["gamma_sigma"] * r[3]
        p = torch.sqrt(gam * gam - 1.0)
        thx, thy = b["divergence"] * r[4], b["divergence"] * r[5]
        u = [p * thx, p * thy, -p * torch.sqrt(1.0 - thx * thx - thy * thy)]
    elif case["op"] == "sweep":
        # 30 lines at the radii (s + 1/2) 0.1 lambda, a 2.6-GeV beam moving along -z
        cfg = workloads.config(6)
        b, s = cfg["beam"], torch.arange(cfg["n_sets"], device="cuda", dtype=torch.float64)
        per = _counts(case, seed)
        x = torch.repeat_interleave((s + 0.5) * cfg["radius_step"], torch.as_tensor(per, device="cuda"))
        y = torch.zeros_like(x)
        z = -case["t0"] + b["sigma_z"] * torch.randn(x.numel(), dtype=torch.float64, device="cuda", generator=g)
        u = [torch.zeros_like(x), torch.zeros_like(x), torch.full_like(x, -math.sqrt(b["gamma"] ** 2 - 1.0))]
    else:
        index = case["workload"] if case["op"] == "push" else 5
        box = workloads.config(index)["box"]
        if index == 4:  # the part of the channel around the moving focus
            zc = 0.99 * (case["t0"] + 0.5 * DT * case["steps"])
            box = box[:2] + ((zc - 40 * L, zc + 40 * L),)
        x, y, z = _uniform(n, box, g)
        u = [torch.zeros_like(x) for _ in range(3)]
    return dict(x=x.contiguous(), y=y.contiguous(), z=z.contiguous(), ux=u[0].to(udt).contiguous(),
                uy=u[1].to(udt).contiguous(), uz=u[2].to(udt).contiguous())


def _counts(case, seed):
    """Particles of each set: log-uniform counts scaled to the case's total
    (batched, adjoint), equal lines (sweep)."""
    if case["op"] == "sweep":
        return np.full(30, max(1, case["n"] // 30), dtype=np.int64)
    s = case["n_sets"]
    r = np.random.RandomState(int(seed) % (1 << 31)).random_sample(s)
    w = np.exp(r * math.log(20.0))
    c = np.maximum(1, np.floor(w * (case["n"] / w.sum()))).astype(np.int64)
    c[0] += max(0, case["n"] - int(c.sum()))
    return c


def _pulses(case, seed):
    """Pulse dicts, one per set."""
    op = case["op"]
    if op == "push":
        return [workloads.config(case["workload"])["pulse"]]
    if op == "sweep":
        return [workloads.config(6)["pulse"]] * 30
    cfg = workloads.config(5)
    r = cfg["ranges"]
    v = np.random.RandomState((int(seed) + 7) % (1 << 31)).random_sample((case["n_sets"], 3))
    v = np.float32(v)  # the adjoint's parameters are float tensors
    out = []
    for a in v:
        d = dict(cfg["pulse"])
        for k, name in enumerate(("a0", "w0", "z_focus")):
            d[name] = float(np.float32(r[name][0] + a[k] * (r[name][1] - r[name][0])))
        out.append(d)
    return out


def _grid(case, seed):
    """Static grid field of workload 2's form on case["grid"]^3 nodes over its box."""
    if not case.get("grid"):
        return None
    cfg = workloads.config(2)
    lo, hi = workloads.grid_box(cfg)
    gk = cfg["grid"]
    return (workloads.grid_field(cfg["box"], case["grid"], gk["amplitude"], gk["n_terms"], gk["kmax"],
                                 seed=int(seed) + 2, torch_device="cuda"), lo, hi)


def _node_pulse(kind):
    if kind == "plane":
        return dict(kind="plane", pol="x", env="gauss", env_len=30.0, a0=1.0)
    if kind == "lg":
        return dict(workloads.config(3)["pulse"], env="gauss", env_len=30.0, t_focus=0.0)
    return workloads.config(2)["pulse"]


def _node_grid(case, seed):
    """Node (0, 0, 0) and the spacings: workload 2's box, shifted by a seeded part of a cell."""
    r = np.random.RandomState(int(seed) % (1 << 31)).random_sample(4)
    ext = (20 * L, 20 * L, 40 * L)
    n = (case["nx"], case["ny"], case["nz"])
    d = [e / k for e, k in zip(ext, n)]
    return [-0.5 * e + s * dd for e, s, dd in zip(ext, r, d)], d, 4.0 * (r[3] - 0.5)


def _line(case, seed):
    """A line's spacing, step, pulse and initial arrays (Sec. 4: lambda/dz = 20,
    dt/dz = 0.9, a super-Gaussian of order 4; the plasma of n_e = 1e-3 n_c with
    a seeded density modulation)."""
    g = _gen(seed)
    dt64 = torch.float64
    dz = L / 20
    dt = 0.9 * dz
    wp = math.sqrt(1e-3)
    pulse = dict(kind="plane", pol="x", env="sgauss", sg_order=4, env_len=30.0, a0=1.0, omega=1.0, omega_p=wp,
                 yee=True, yee_dx=dz, yee_dt=dt)
    nl, nz = case["n_lines"], case["nz"]
    z0 = -0.5 * nz * dz
    k = torch.arange(nz, dtype=dt64, device="cuda")
    ph = 2 * math.pi * torch.rand((nl, 1), dtype=dt64, device="cuda", generator=g)
    wp2 = wp * wp * (1.0 + 0.1 * torch.cos(2 * math.pi * 3 * k[None, :] / nz + ph))
    amp = 1.0 + 0.1 * torch.rand((nl, 1), dtype=dt64, device="cuda", generator=g)
    if case["form"] == "split":
        E = torch.zeros((nl, nz), dtype=dt64, device="cuda")
        B = torch.zeros_like(E)
        J = 1e-3 * amp * torch.exp(-(((z0 + k * dz) / 30.0) ** 8))[None, :] * torch.sin(z0 + k * dz)[None, :]
    else:
        env = torch.exp(-(((z0 + k * dz) / 30.0) ** 8))[None, :]
        E = amp * env * torch.cos(z0 + k * dz)[None, :]
        B = amp * env * torch.cos(z0 + (k + 0.5) * dz)[None, :]
        J = torch.zeros_like(E)
    td = getattr(torch, case["dtype"])
    arr = {n: v.to(td).contiguous() for n, v in dict(E=E, B=B, J=J, wp2=wp2).items()}
    return dict(dz=dz, dt=dt, z0=z0, pulse=pulse, arr=arr)


# ---------------------------------------------------------------- prepare, run

# the shapes the autotuner picks for the workloads on this GPU
_TUNED = {("push", 2, True): dict(block=256, grid_cache=2, pairs=1), ("push", 2, False): dict(block=128, pairs=1),
          ("push", 1, False): dict(block=128, pairs=1), ("push", 3, False): dict(block=256, pairs=1),
          ("push", 4, False): dict(block=128, pairs=1), ("batch", 0, False): dict(block=64, pairs=1, tile=256),
          ("sweep", 0, False): dict(block=64, pairs=1, tile=128)}


def prepare(case, seed):
    op = case["op"]
    s = dict(case=case)
    if op in ("push", "batch", "sweep"):
        s["init"] = _ensemble(case, seed)
        s["work"] = {k: v.clone() for k, v in s["init"].items()}
        s["h"] = _lib.Handle(_pulses(case, seed))
        grid = _grid(case, seed)
        s["grid"] = _lib.pack_grid(grid, layout="cells") if grid is not None else None
        if case["launch"] == "tuned":
            s["h"].set_launch(**_TUNED[op, case.get("workload", 0), bool(case.get("grid"))])
        s["t"] = case["t0"]
        s["diag"] = None
        if case.get("lightfront"):
            s["diag"] = dict(lightfront=torch.zeros(case["steps"], dtype=torch.float64, device="cuda"))
        if op != "push":
            c = _counts(case, seed)
            s["off"] = torch.as_tensor(np.concatenate([[0], np.cumsum(c)]).astype(np.int64)).cuda()
            s["count"] = torch.as_tensor(c, dtype=torch.float64).cuda()
            s["diag"] = dict(set_sum=torch.zeros(len(c), dtype=torch.float64, device="cuda"))
            s["ws"] = torch.zeros(_lib.ap_batch_workspace_bytes(s["h"].h) // 4, dtype=torch.int32, device="cuda")
            if case.get("graph"):
                st = torch.cuda.Stream()
                st.wait_stream(torch.cuda.current_stream())
                s["graph"] = _lib.ap_batch_graph_create(s["h"].h, s["work"], s["off"], None, case["t0"], DT,
                                                        case["steps"], "fp32", s["diag"], s["ws"], st)
    elif op == "adjoint":
        s["parts"] = _ensemble(case, seed)
        s["pulses"] = _pulses(case, seed)
        s["off"] = torch.as_tensor(np.concatenate([[0], np.cumsum(_counts(case, seed))]).astype(np.int64)).cuda()
        s["params"] = torch.tensor([[d["a0"], d["w0"], d["z_focus"]] for d in s["pulses"]], dtype=torch.float32,
                                   device="cuda", requires_grad=True)
    elif op == "nodes":
        s["h"] = _lib.Handle(_node_pulse(case["kind"]))
        s["lo"], s["d"], s["t"] = _node_grid(case, seed)
        shape = (6, case["nz"], case["ny"], case["nx"])
        dtype = getattr(torch, case["dtype"])
        if case["accumulate"]:
            s["base"] = 0.1 * torch.randn(shape, dtype=dtype, device="cuda", generator=_gen(seed))
        s["f"] = torch.empty(shape, dtype=dtype, device="cuda")
    elif op == "line":
        s.update(_line(case, seed))
        s["work"] = {k: s["arr"][k].clone() for k in ("E", "B", "J")}
        s["h"] = _lib.Handle(s["pulse"]) if case["form"] == "split" else None
    else:
        g = torch.randn((6, case["nz"], case["ny"], case["nx"]), dtype=torch.float32, device="cuda", generator=_gen(seed))
        s["grid"] = (0.1 * g, (-1.0, -1.0, -1.0), (1.0, 1.0, 1.0))
        cells = (case["nx"] - 1) * (case["ny"] - 1) * (case["nz"] - 1)
        nodes = case["nx"] * case["ny"] * case["nz"]
        s["packed"] = torch.empty(48 * cells if case["layout"] == "cells" else 8 * nodes, dtype=torch.float32, device="cuda")
    return s


_STATE = ("x", "y", "z", "ux", "uy", "uz")


def _restore(s):
    keys = list(s["work"])
    torch._foreach_copy_([s["work"][k] for k in keys], [s["init" if "init" in s else "arr"][k] for k in keys])


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "push":
        if case.get("loop"):  # a step of the caller's own loop: the state moves on in place
            s["h"].push(s["work"], s["t"], DT, case["steps"], precision=case["precision"], grid=s["grid"])
            s["t"] += DT * case["steps"]
            return s["work"]
        _restore(s)
        s["h"].push(s["work"], case["t0"], DT, case["steps"], precision=case["precision"], grid=s["grid"], diag=s["diag"])
        if case["precision"] == "fp64":
            return dict(s["work"], **({"lightfront": s["diag"]["lightfront"]} if s["diag"] else {}))
        return {k: s["work"][k].float() for k in _STATE}
    if op in ("batch", "sweep"):
        _restore(s)
        if "graph" in s:
            _lib.ap_graph_launch(s["graph"])
        else:
            _lib.ap_gather_push_batched(s["h"].h, s["work"], s["off"], None, case["t0"], DT, case["steps"], "fp32",
                                        s["diag"], s["ws"])
        out = {k: s["work"][k].float() for k in _STATE}
        out["mean_gamma"] = (s["diag"]["set_sum"] / s["count"]).float()
        return out
    if op == "adjoint":
        s["params"].grad = None
        J = autograd.mean_final_gamma(s["params"], s["pulses"], s["parts"], s["off"], case["t0"], DT, case["steps"],
                                      case["ckpt"], "fp32")
        J.sum().backward()
        return dict(J=J.detach(), grad=s["params"].grad)
    if op == "nodes":
        if case["accumulate"]:
            s["f"].copy_(s["base"])
        s["h"].eval_nodes(list(s["f"]), s["lo"], s["d"], s["t"], accumulate=case["accumulate"], precision=case["precision"])
        return s["f"]
    if op == "line":
        _restore(s)
        w = s["work"]
        if case["form"] == "split":
            s["h"].apt1d(w["E"], w["B"], w["J"], s["z0"], s["dz"], 0.0, s["dt"], case["steps"], wp2=s["arr"]["wp2"])
        elif case["form"] == "plasma":
            _lib.ap_plasma1d_run(w["E"], w["B"], w["J"], s["dz"], s["dt"], case["steps"], wp2=s["arr"]["wp2"])
        else:
            _lib.ap_yee1d_run(w["E"], w["B"], s["dz"], s["dt"], case["steps"])
            return dict(E=w["E"], B=w["B"])
        return dict(w)
    _lib.ap_grid_pack(s["grid"], s["packed"], layout=case["layout"])
    return s["packed"]


# ------------------------------------------------------------------------ work

def work(case):
    """Bytes and floating-point operations of one pass (an FMA is two): each
    input read once and each output written once; operations counted from the
    formulas."""
    op = case["op"]
    if op in ("push", "batch", "sweep"):
        # one particle-step: field evaluation, Boris step and position update
        per = {1: 100, 2: 190, 3: 290, 4: 3500}[case["workload"]] if op == "push" else 190
        per += 100 if case.get("grid") else 0
        b = 2 * (48 if case.get("precision") == "fp64" else 36) * case["n"]
        b += 192 * max(0, case.get("grid", 0) - 1) ** 3
        return dict(bytes=b, flops=per * case["n"] * case["steps"])
    if op == "adjoint":
        return dict(bytes=36 * case["n"], flops=850 * case["n"] * case["steps"])
    if op == "nodes":
        n = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=(48 if case["accumulate"] else 24) * n, flops=(6 if case["kind"] == "plane" else 150) * n)
    if op == "line":
        n = case["n_lines"] * case["nz"]
        per = {"split": 90, "plasma": 12, "yee": 9}[case["form"]]
        return dict(bytes={"split": 28, "plasma": 28, "yee": 16}[case["form"]] * n, flops=per * n * case["steps"])
    nodes = case["nx"] * case["ny"] * case["nz"]
    cells = (case["nx"] - 1) * (case["ny"] - 1) * (case["nz"] - 1)
    if case["layout"] == "nodes":
        return dict(bytes=(24 + 32) * nodes, flops=0)
    return dict(bytes=24 * nodes + 192 * cells, flops=6 * 19 * cells)


# ----------------------------------------------------------- the same in 64 bits

_POL = {"x": (1, 0), "y": (0, 1), "cp": (1, -1j), "cm": (1, 1j)}


def _envelope(d, eta):
    env = d.get("env", "cw")
    if env == "sin2":
        T = 2 * math.pi * d["env_len"] / d.get("omega", 1.0)
        return torch.where(eta.abs() <= 0.5 * T, torch.cos(math.pi * eta / T) ** 2, torch.zeros_like(eta))
    if env == "gauss":
        return torch.exp(-2 * math.log(2.0) * (eta / d["env_len"]) ** 2)
    if env == "sgauss":
        return torch.exp(-((eta / d["env_len"]) ** (2 * d["sg_order"])))
    return torch.ones_like(eta)


def _laguerre(p, a, s):
    lm, lp = torch.zeros_like(s), torch.ones_like(s)
    for k in range(p):
        lm, lp = lp, ((2 * k + 1 + a - s) * lp - (k + a) * lm) / (k + 1)
    return lp


def _lg_norm(p, a):
    """max over s of s^(a/2) |L_p^a(s)| exp(-s/2), from the roots of its derivative."""
    c = [(-1) ** i * math.comb(p + a, p - i) / math.factorial(i) for i in range(p + 1)]
    P = np.polynomial.Polynomial(c)
    S = np.polynomial.Polynomial([0.0, 1.0])
    r = (0.5 * a * P + S * P.deriv() - 0.5 * S * P).roots()
    r = np.array([0.0] + [v.real for v in r if abs(v.imag) < 1e-9 and v.real > 0])
    return float(np.max(r ** (0.5 * a) * np.abs(P(r)) * np.exp(-0.5 * r)))


def _flying_table(d):
    n = d["n_comp"]
    f = np.arange(n) / (n - 1)
    w = 1.0 - d["bw_frac"] + 2 * d["bw_frac"] * f
    zj = d["z_focus"] + d["ff_length"] * f
    tau = d["t_focus"] + (zj - d["z_focus"]) / d["beta_f"] - zj
    zR = 0.5 * w * d["w0"] ** 2
    Phi = np.concatenate([[0.0], np.cumsum(0.5 * (tau[1:] + tau[:-1]) * (w[1:] - w[:-1]))])
    zm, tm = d["z_focus"] + 0.5 * d["ff_length"], d["t_focus"] + 0.5 * d["ff_length"] / d["beta_f"]
    z = zm - 0.25 * d["ff_length"] + 0.5 * d["ff_length"] * np.arange(2049) / 2048
    S = sum(np.exp(1j * (w[j] * (tm - z) - Phi[j])) / (1 - 1j * (z - zj[j]) / zR[j]) for j in range(n))
    return w, zj, zR, Phi, d["a0"] / np.max(np.abs(S))


def _field(d, x, y, z, t):
    """E1, B1 (lists of three) of a vacuum pulse in 64 bits; pulse parameters may
    be one value or one per particle."""
    px, py = _POL[d.get("pol", "x")]
    kind = d.get("kind", "plane")
    T, dz = t - d.get("t_focus", 0.0), z - d.get("z_focus", 0.0)
    if kind == "flying":
        w, zj, zR, Phi, A = _flying_table(d)
        r2 = x * x + y * y
        U, W = torch.zeros_like(x, dtype=torch.complex128), torch.zeros_like(x, dtype=torch.complex128)
        for j in range(d["n_comp"]):
            q = 1.0 / torch.complex(torch.ones_like(z), -(z - zj[j]) / zR[j])
            a = (-r2 / d["w0"] ** 2) * q
            Uj = A * q * torch.exp(torch.complex(a.real, a.imag + w[j] * (t - z) - Phi[j]))
            U, W = U + Uj, W + q * Uj / w[j]
        g = -2.0 / d["w0"] ** 2
        dUx, dUy, lon = g * x * W, g * y * W, 1.0
    else:
        psi = T - dz + d.get("phase0", 0.0)
        amp = d["a0"] * _envelope(d, T - dz)
        if kind == "plane":
            U = torch.complex(amp * torch.cos(psi), amp * torch.sin(psi))
            dUx = dUy = None
        else:
            zeta = dz / (0.5 * d["w0"] ** 2)
            q = 1.0 / torch.complex(torch.ones_like(zeta), -zeta)
            iw = 1.0 / d["w0"] ** 2
            a = (-(x * x + y * y) * iw) * q
            base = amp * torch.exp(torch.complex(a.real, a.imag + psi))
            if kind == "gauss":
                U = base * q
                dUx, dUy = -2 * iw * x * q * U, -2 * iw * y * q * U
            else:
                p, l = d["lg_p"], d["lg_l"]
                al, sg = abs(l), 1.0 if l >= 0 else -1.0
                s = 2 * (x * x + y * y) * iw * q.real
                Lp = _laguerre(p, al, s)
                dL = -_laguerre(p - 1, al + 1, s) if p > 0 else torch.zeros_like(s)
                xi = torch.complex(x, sg * y)
                K = base * (q ** (al + 1)) * (q / q.conj()) ** p * ((math.sqrt(2.0) / d["w0"]) ** al / _lg_norm(p, al))
                xa = xi ** al
                U = K * xa * Lp
                T1 = al * xi ** (al - 1) * Lp if al else torch.zeros_like(U)
                T2 = xa * (4 * q.real * iw * dL - 2 * iw * Lp * q)
                dUx, dUy = K * (T1 + x * T2), K * (1j * sg * T1 + y * T2)
        lon = 1.0
    zero = torch.zeros_like(x)
    E, B = [(px * U).real, (py * U).real, zero], [-(py * U).real, (px * U).real, zero]
    if d.get("longitudinal") and dUx is not None:
        E[2] = lon * (px * dUx + py * dUy).imag
        B[2] = lon * (-py * dUx + px * dUy).imag
    return E, B


def _gather(grid, x, y, z):
    f, lo, hi = grid
    w, i0 = [], []
    for v, a, n in ((x, 0, f.shape[3]), (y, 1, f.shape[2]), (z, 2, f.shape[1])):
        u = ((v - lo[a]) * ((n - 1) / (hi[a] - lo[a]))).clamp(0, n - 1)
        i = u.floor().clamp(max=n - 2)
        w.append(u - i)
        i0.append(i.long())
    nx, ny = f.shape[3], f.shape[2]
    flat = f.reshape(6, -1)
    out = [0.0] * 6
    for c in range(8):
        b = (c & 1, (c >> 1) & 1, c >> 2)
        at = ((i0[2] + b[2]) * ny + i0[1] + b[1]) * nx + i0[0] + b[0]
        ww = (w[0] if b[0] else 1 - w[0]) * (w[1] if b[1] else 1 - w[1]) * (w[2] if b[2] else 1 - w[2])
        for k in range(6):
            out[k] = out[k] + ww * flat[k][at].double()
    return out


def _step(d, p, t, grid=None):
    """One step of the push on p = [x, y, z, ux, uy, uz]."""
    x, y, z = p[:3]
    E, B = _field(d, x, y, z, t)
    if grid is not None:
        G = _gather(grid, x, y, z)
        E, B = [a + b for a, b in zip(E, G[:3])], [a + b for a, b in zip(B, G[3:])]
    h = -0.5 * DT
    m = [u + h * e for u, e in zip(p[3:], E)]
    ig = torch.rsqrt(1 + m[0] * m[0] + m[1] * m[1] + m[2] * m[2])
    tau = [h * ig * b for b in B]
    f = 2 / (1 + tau[0] * tau[0] + tau[1] * tau[1] + tau[2] * tau[2])

    def cross(a, b):
        return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]

    q = [a + c for a, c in zip(m, cross(m, tau))]
    q = [a + f * c for a, c in zip(m, cross(q, tau))]
    u = [a + h * e for a, e in zip(q, E)]
    ig = torch.rsqrt(1 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
    dxy = 0.0 if d.get("one_d") else DT
    return [x + dxy * u[0] * ig, y + dxy * u[1] * ig, z + DT * u[2] * ig] + u


def _per_particle(case, seed):
    """The pulse of every particle (one value per particle where the sets differ)."""
    ps = _pulses(case, seed)
    d = dict(ps[0])
    if case["op"] in ("batch", "adjoint"):
        idx = torch.repeat_interleave(torch.arange(len(ps), device="cuda"), torch.as_tensor(_counts(case, seed), device="cuda"))
        for k in ("a0", "w0", "z_focus"):
            d[k] = torch.tensor([p[k] for p in ps], dtype=torch.float64, device="cuda")[idx]
        return d, idx
    return d, None


def _exact_push(case, seed):
    parts = _ensemble(case, seed)
    p = [parts[k].double() for k in _STATE]
    d, idx = _per_particle(case, seed)
    grid = _grid(case, seed)
    h0 = torch.sqrt(1 + p[3] ** 2 + p[4] ** 2 + p[5] ** 2) - p[5]
    lf = []
    for n in range(case["steps"]):
        p = _step(d, p, case["t0"] + n * DT, grid)
        if case.get("lightfront"):
            lf.append((torch.sqrt(1 + p[3] ** 2 + p[4] ** 2 + p[5] ** 2) - p[5] - h0).abs().max())
    out = dict(zip(_STATE, p))
    if case.get("lightfront"):
        out["lightfront"] = torch.stack(lf)
    if case["op"] in ("batch", "sweep"):
        c = torch.as_tensor(_counts(case, seed), device="cuda")
        idx = torch.repeat_interleave(torch.arange(len(c), device="cuda"), c)
        g = torch.sqrt(1 + p[3] ** 2 + p[4] ** 2 + p[5] ** 2)
        out["mean_gamma"] = torch.zeros(len(c), dtype=torch.float64, device="cuda").index_add_(0, idx, g) / c
    return out


def _exact_adjoint(case, seed):
    """Mean final gammas and their gradients: segments of ten steps, each run
    again under autograd on the way back."""
    parts = _ensemble(case, seed)
    p = [parts[k].double() for k in _STATE]
    d, idx = _per_particle(case, seed)
    c = torch.as_tensor(_counts(case, seed), device="cuda", dtype=torch.float64)
    par = torch.tensor([[q["a0"], q["w0"], q["z_focus"]] for q in _pulses(case, seed)], dtype=torch.float64, device="cuda")
    seg, saved = 10, []
    with torch.no_grad():
        for n in range(case["steps"]):
            if n % seg == 0:
                saved.append(p)
            p = _step(d, p, case["t0"] + n * DT)
        g = torch.sqrt(1 + p[3] ** 2 + p[4] ** 2 + p[5] ** 2)
        J = torch.zeros_like(c).index_add_(0, idx, g) / c
        wt = 1.0 / (g * c[idx])
        lam = [torch.zeros_like(g) for _ in range(3)] + [u * wt for u in p[3:]]
    grad = torch.zeros_like(par)
    for k in range(len(saved) - 1, -1, -1):
        q = [v.detach().requires_grad_() for v in saved[k]]
        pr = par.clone().requires_grad_()
        dd = dict(d)
        for j, name in enumerate(("a0", "w0", "z_focus")):
            dd[name] = pr[:, j][idx]
        o = q
        for n in range(k * seg, min(case["steps"], (k + 1) * seg)):
            o = _step(dd, o, case["t0"] + n * DT)
        got = torch.autograd.grad(o, q + [pr], lam)
        lam = list(got[:6])
        grad += got[6]
        saved[k] = None
    return dict(J=J, grad=grad)


def _exact_nodes(case, seed):
    d = _node_pulse(case["kind"])
    lo, dd, t = _node_grid(case, seed)
    n = (case["nx"], case["ny"], case["nz"])
    off = ((1, 0, 0), (0, 1, 0), (0, 0, 1), (0, 1, 1), (1, 0, 1), (1, 1, 0))
    shape = (6, n[2], n[1], n[0])
    out = torch.empty(shape, dtype=torch.float64, device="cuda")
    for c in range(6):
        ax = [lo[a] + (torch.arange(n[a], dtype=torch.float64, device="cuda") + 0.5 * off[c][a]) * dd[a] for a in range(3)]
        for k in range(0, n[2], 32):
            z, y, x = torch.meshgrid(ax[2][k:k + 32], ax[1], ax[0], indexing="ij")
            E, B = _field(d, x, y, z, t)
            out[c, k:k + 32] = (E + B)[c]
    if case["accumulate"]:
        out += 0.1 * torch.randn(shape, dtype=getattr(torch, case["dtype"]), device="cuda", generator=_gen(seed))
    return out


def _exact_line(case, seed):
    s = _line(case, seed)
    E, B, J, wp2 = (s["arr"][k].double().clone() for k in ("E", "B", "J", "wp2"))
    dz, dt, d = s["dz"], s["dt"], s["pulse"]
    r = dt / dz
    if case["form"] == "yee":
        wp2 = torch.zeros_like(wp2)
    split = case["form"] == "split"
    if split:
        # exact discrete dispersion of the Yee line with the leapfrog current (Sec. 4)
        wp = d["omega_p"]
        h, q = 0.5 * dt, 0.5 * wp * dt
        s2 = (math.sin(h) ** 2 - q * q) / (r * r)
        k = 2 * math.asin(math.sqrt(s2)) / dz
        vg = r * r * math.sqrt(s2 * (1 - s2)) * dz / (math.sin(h) * math.cos(h) * dt)
        jamp = wp * wp * (h / math.sin(h))
        zk = s["z0"] + dz * torch.arange(case["nz"], dtype=torch.float64, device="cuda")
        g2, tau = 2 * d["sg_order"], d["env_len"]
    for n in range(case["steps"]):
        B[:, :-1] -= 0.5 * r * (E[:, 1:] - E[:, :-1])
        drive, J1 = E, 0.0
        if split:
            t = n * dt
            drive = E + d["a0"] * torch.exp(-(((t - zk / vg) / tau) ** g2)) * torch.cos(t - k * zk)
            t += 0.5 * dt
            u = (t - zk / vg) / tau
            L1 = -(g2 / tau) * u ** (g2 - 1)
            L2 = L1 * L1 - g2 * (g2 - 1) / tau ** 2 * u ** (g2 - 2)
            J1 = (jamp * d["a0"]) * torch.exp(-(u ** g2)) * (1 - L2 + 0.5 * L1 * L1) * torch.sin(t - k * zk + L1)
        J += dt * wp2 * drive
        src = (J - J1)[:, 1:]
        E[:, 1:] -= r * (B[:, 1:] - B[:, :-1]) + dt * src
        B[:, :-1] -= 0.5 * r * (E[:, 1:] - E[:, :-1])
    return dict(E=E, B=B, J=J) if case["form"] != "yee" else dict(E=E, B=B)


def _exact_pack(case, seed):
    f = prepare(case, seed)["grid"][0].double()
    if case["layout"] == "nodes":
        out = torch.zeros(f.shape[1:] + (8,), dtype=torch.float64, device="cuda")
        out[..., :6] = f.permute(1, 2, 3, 0)
        return out.reshape(-1)
    c = {(i, j, k): f[:, k:f.shape[1] - 1 + k, j:f.shape[2] - 1 + j, i:f.shape[3] - 1 + i]
         for i in (0, 1) for j in (0, 1) for k in (0, 1)}
    a1, a2, a3 = c[1, 0, 0] - c[0, 0, 0], c[0, 1, 0] - c[0, 0, 0], c[0, 0, 1] - c[0, 0, 0]
    a4 = c[1, 1, 0] - c[1, 0, 0] - a2
    a5 = c[0, 1, 1] - c[0, 1, 0] - a3
    a6 = c[1, 0, 1] - c[1, 0, 0] - a3
    a7 = (c[1, 1, 1] - c[1, 1, 0] - (c[1, 0, 1] - c[1, 0, 0])) - a5
    out = torch.stack([c[0, 0, 0], a1, a2, a3, a4, a5, a6, a7], dim=-1)  # [6, z, y, x, 8]
    # components in pairs, both components of a coefficient side by side
    out = out.reshape((3, 2) + out.shape[1:]).permute(2, 3, 4, 0, 5, 1)
    return out.reshape(-1)


def exact(case, seed):
    with torch.no_grad():
        op = case["op"]
        if op in ("push", "batch", "sweep"):
            return _exact_push(case, seed)
        if op == "nodes":
            return _exact_nodes(case, seed)
        if op == "line":
            return _exact_line(case, seed)
        if op == "pack":
            return _exact_pack(case, seed)
    return _exact_adjoint(case, seed)

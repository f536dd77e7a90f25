"""The performance cases: what a user of this library has it do, through its public entry
points (paper_2506_16076_gb300.fcsdnn), from one small shock tube to the 28M-point Mach-25
array.

A case is a dict of plain values: `op` (the entry point), `kind` (the patch layout), its
sizes and options. Every state is a flow with a compressed layer behind a smeared front
(radius or position from the seed), a no-slip layer at a body and a smooth perturbation, so
that some lines carry viscosity and most do not, as in a run.

  rhs      Context.rhs, one evaluation of the operator with the viscosity given
  noalloc  rhs_patch_noalloc, the same for one stand-alone patch and no allocation
  filter   Context.filter, the per-step spectral filter
  visc     Context.viscosity and Context.timestep: what a step needs besides its stages
  step     Context.rk_step, a whole filtered time step from a stored state (as a checkpoint
           replay does), captured as a CUDA graph
  host     Context.rk_step_host, the same with the state in page-locked host memory
  adjoint  Context.adjoint_step of a filtered step, gradients with respect to the state, the
           Dirichlet data, the Mach number and the angle of attack
"""
import dataclasses
import math
import os

import numpy as np
import torch

from paper_2506_16076_gb300 import fcsdnn as F
from paper_2506_16076_gb300 import workloads as W

GAMMA = 1.4


def listed():
    return [
        # the 128 x 128 shock tube of the test suite: the smallest calls, bound by latency
        {"name": "rhs_sod128", "op": "rhs", "kind": "box", "n1": 128, "n2": 128, "policy": 0},
        {"name": "step_sod128", "op": "step", "kind": "box", "n1": 128, "n2": 128, "policy": 0},
        # one ragged patch as large as the longest lines of the seeded arrays, cheap continuation
        {"name": "rhs_box_ragged", "op": "rhs", "kind": "box", "n1": 509, "n2": 333, "policy": 2},
        # the stand-alone entry at its size limit per patch, for callers that own all memory
        {"name": "noalloc_485", "op": "noalloc", "kind": "box", "n1": 485, "n2": 485, "policy": 0},
        # the Mach-3 cylinder (0.46M points): the ordinary multi-patch run and its passes
        {"name": "step_cyl_m3", "op": "step", "kind": "cyl", "scale": 1.0},
        {"name": "filter_cyl_m3", "op": "filter", "kind": "cyl", "scale": 1.0},
        # the same with the state handed over in host memory every step
        {"name": "host_cyl_m3", "op": "host", "kind": "cyl", "scale": 1.0},
        # the cylinder on S-type arcs: curvilinear lines, product-rule wall form
        {"name": "rhs_cyl_m3_stype", "op": "rhs", "kind": "stype", "wall_form": 1},
        # the adjoint configuration (Mach 2 at 2 degrees), and a larger seeded array
        {"name": "adjoint_cyl_m2_half", "op": "adjoint", "kind": "half"},
        {"name": "adjoint_array8", "op": "adjoint", "kind": "array", "nx": 8, "nmax": 384, "seed": 3},
        # viscosity and time step of a quarter of the Mach-25 array's patches
        {"name": "visc_array16", "op": "visc", "kind": "array", "nx": 16, "nmax": 384, "seed": 3},
        # the 32 x 32 seeded array at Mach 25 (28M points), the headline workload
        {"name": "step_cyl_m25_32", "op": "step", "kind": "array", "nx": 32, "nmax": 384, "seed": 3},
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    op = rng.choice(["rhs", "rhs", "step", "step", "filter", "visc", "adjoint", "host", "noalloc"])
    if op == "noalloc":  # its limits: 262144 points, 997 per line
        n1 = _log(rng, 32, 900)
        return {"op": op, "kind": "box", "n1": n1, "n2": _log(rng, 32, min(900, 262144 // n1)), "policy": 0}
    kind = rng.choice(["box", "box", "cyl", "array", "array", "stype" if op == "rhs" else "half"])
    if kind == "box":
        return {"op": op, "kind": kind, "n1": _log(rng, 40, 1200), "n2": _log(rng, 40, 1200), "policy": rng.choice([1, 2, 2])}
    if kind == "cyl":
        return {"op": op, "kind": kind, "scale": round(rng.uniform(0.6, 2.0), 3)}
    if kind == "stype":
        return {"op": op, "kind": kind, "wall_form": rng.choice([0, 1]), "half": rng.choice([8, 10, 12])}
    if kind == "half":
        return {"op": op, "kind": kind, "mach": round(rng.uniform(1.6, 3.2), 3)}
    return {"op": op, "kind": kind, "nx": rng.choice([4, 6, 8, 10, 12, 16]), "nmax": rng.randint(300, 384), "seed": rng.randrange(1, 1000)}


def workload(case):
    k = case["kind"]
    if k == "box":
        w = W.sod128()
        n1, n2 = case["n1"], case["n2"]
        p = dataclasses.replace(w.patches[0], n1=n1, n2=n2, geom=(0.0, 1.0, 0.0, (n2 - 1) / (n1 - 1)))
        return dataclasses.replace(w, name=f"box{n1}x{n2}", patches=[p], params=dataclasses.replace(w.params, c_policy=case["policy"]))
    if k == "cyl":
        return W.cyl_m3(case["scale"])
    if k == "half":
        return W.cyl_m2_half(mach=case.get("mach", 2.0))
    if k == "stype":
        w = W.cyl_m3_stype(half=case.get("half", 8))
        return dataclasses.replace(w, params=dataclasses.replace(w.params, wall_form=case["wall_form"]))
    return W.cyl_m25_array(case["nx"], 48, case["nmax"], case["seed"], 0.6, 1024, 192, "array")


def _xy(w):
    """Coordinates of all points on the GPU, patch after patch."""
    X, Y = [], []
    for p in w.patches:
        if p.kind == W.AFFINE:  # the box's two axes go over, the grid is made there
            x0, x1, y0, y1 = p.geom
            x = torch.linspace(x0, x1, p.n1, dtype=torch.float64, device="cuda")
            y = torch.linspace(y0, y1, p.n2, dtype=torch.float64, device="cuda")
            X.append(x.expand(p.n2, p.n1).reshape(-1))
            Y.append(y[:, None].expand(p.n2, p.n1).reshape(-1))
        else:
            for out, a in zip((X, Y), W.patch_xy(p)):
                out.append(torch.from_numpy(np.ascontiguousarray(a)).cuda().reshape(-1))
    return torch.cat(X), torch.cat(Y)


def _flow(case, w, seed):
    """(state [4][P], viscosity [P]) from the seed."""
    r = np.random.default_rng(seed)
    x, y = _xy(w)
    rho0, u0, v0, p0 = w.freestream
    if case["kind"] == "box":
        at = 0.35 + 0.3 * r.random()
        dist = x - at - 0.05 * torch.sin(3.0 * y)
        width, body = 0.02, torch.ones_like(x)
        u0 = 0.5
    else:
        rad = torch.hypot(x, y)
        at = 1.9 + 0.8 * r.random()
        dist = torch.hypot(x - 0.4, y) - at
        width, body = 0.08, 1.0 - torch.exp(-(((rad - 0.5).clamp(min=0.0) / 0.1) ** 2))
    s = 0.5 * (1.0 - torch.tanh(dist / width))
    k, ph = r.uniform(0.5, 2.0, 4), r.uniform(0.0, 2.0 * np.pi, 4)
    q = [0.02 * torch.sin(k[c] * x + ph[c]) * torch.cos(k[c] * y + 0.3 * ph[c]) for c in range(4)]
    rho = rho0 * (1.0 + 1.5 * s) * (1.0 + q[0])
    u = body * (u0 * (1.0 - 0.5 * s) + q[1])
    v = body * (v0 + q[2])
    p = p0 * (1.0 + 4.0 * s) * (1.0 + q[3])
    e = torch.stack([rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)]).contiguous()
    mu = 0.01 * (1.0 - (dist / (4.0 * width)) ** 2).clamp(min=0.0)
    return e, mu


def prepare(case, seed):
    w = workload(case)
    e, mu = _flow(case, w, seed)
    s = {"op": case["op"], "e": e, "mu": mu}
    if case["op"] == "noalloc":
        p = w.patches[0]
        s |= {"out": torch.empty_like(e), "n": (p.n1, p.n2), "box": p.geom}
        return s
    s["ctx"] = ctx = F.Context(w)
    s["dt"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    if case["op"] == "rhs":
        s["out"] = torch.empty_like(e)
    elif case["op"] in ("step", "filter"):
        s["now"] = torch.empty_like(e)
    elif case["op"] == "host":
        s["e"] = e.cpu().pin_memory()
        s["now"] = torch.empty_like(s["e"]).pin_memory()
    elif case["op"] == "adjoint":
        ctx.project(e)
        ctx.timestep(e, mu, s["dt"])
        g = torch.Generator(device="cuda").manual_seed(seed)
        s["lam"] = torch.randn(e.shape, dtype=torch.float64, device="cuda", generator=g)
        s |= {"out": torch.empty_like(e), "gbc": torch.zeros_like(e), "dpar": torch.zeros(2, dtype=torch.float64, device="cuda")}
    # a user's program marches on a stream of its own: a graph is not captured on the default one
    s["stream"] = torch.cuda.Stream()
    s["stream"].wait_stream(torch.cuda.current_stream())
    return s


def run(s):
    op = s["op"]
    if op == "noalloc":
        F.rhs_patch_noalloc(s["e"], s["mu"], s["out"], *s["n"], s["box"], 5, 27)
        return s["out"]
    ctx, st = s["ctx"], s["stream"]
    with torch.cuda.stream(st):
        if op == "rhs":
            ctx.rhs(s["e"], s["out"], s["mu"])
            return s["out"]
        if op == "filter":
            s["now"].copy_(s["e"])
            ctx.filter(s["now"])
            return s["now"]
        if op == "visc":
            ctx.viscosity(s["e"], s["mu"])
            ctx.timestep(s["e"], s["mu"], s["dt"])
            return s["mu"], s["dt"]
        if op == "step":
            s["now"].copy_(s["e"])
            ctx.rk_step(s["now"], s["dt"], s["mu"], F.STEP_FILTER | F.STEP_GRAPH)
            return s["now"], s["mu"], s["dt"]
        if op == "host":
            s["now"].copy_(s["e"])
            ctx.rk_step_host(s["now"], s["dt"], s["mu"], F.STEP_FILTER | F.STEP_GRAPH)
            return s["now"], s["mu"], s["dt"]
        s["gbc"].zero_()
        s["dpar"].zero_()
        ctx.adjoint_step(s["e"], s["mu"], s["dt"], s["lam"], s["out"], s["gbc"], F.STEP_FILTER,
                         s["dpar"] if s["ctx"].w.freestream[1] > 0 else None)
        return s["out"], s["gbc"], s["dpar"]


def work(case):
    """State-sized reads and writes of the call, and the FP64 flops of its FC lines (a real FFT
    pair of 5 n log2 n flops per line and component) and pointwise work."""
    w = workload(case)
    pts = sum(p.npts for p in w.patches)
    line = sum(p.npts * 2.5 * (math.log2(p.n1) + math.log2(p.n2)) for p in w.patches) * 2.0  # per component, both directions
    rhs = 2.0 * 4.0 * line + 80.0 * pts  # gradient and divergence rounds
    filt = 4.0 * line + 20.0 * pts
    visc = 400.0 * pts
    by, fl = {"rhs": (9, rhs), "noalloc": (9, rhs), "filter": (8, filt), "visc": (5, visc), "step": (9, 5 * rhs + filt + visc),
              "host": (9, 5 * rhs + filt + visc), "adjoint": (17, 15 * rhs + 2 * filt)}[case["op"]]
    return {"bytes": 8.0 * by * pts, "flops": fl}


# ---- 64-bit values of the operator and the filter on one box, by the method's definition

def _tables(d):
    """C -> (A_l Q^T, A_r Q^T) of the FC-Gram data file of order d."""
    path = os.path.join(os.path.dirname(os.path.abspath(F.__file__)), "data", f"fc_tables_d{d}.txt")
    out, rows, name = {}, None, None
    with open(path) as f:
        for t in (ln.split() for ln in f):
            if not t or t[0].startswith("#"):
                continue
            if t[0] == "C":
                rows = out[int(t[1])] = {}
            elif t[0] in ("Q", "AL", "AR"):
                name = t[0]
                rows[name] = []
            elif not t[0][0].isalpha():
                rows[name].append([np.longdouble(v) for v in t])
    return {c: tuple(np.array(r[a]) @ np.array(r["Q"]).T for a in ("AL", "AR")) for c, r in out.items()}


def _lines(f, C, tab, mult):
    """FC lines along the last axis: continue, transform, multiply by mult(k, L), transform back."""
    d, n = 5, f.shape[-1]
    ML, MR = tab[C]
    ext = f[..., :d] @ ML.T + f[..., n - d:] @ MR.T
    c = np.concatenate([f, ext], axis=-1)
    L = c.shape[-1]
    k = np.fft.fftfreq(L, 1.0 / L).round().astype(np.longdouble)
    return np.fft.ifft(mult(k, L) * np.fft.fft(c, axis=-1), axis=-1).real[..., :n]


def _cost(L):
    """Transform cost estimate that rules the cheap continuation (policy 2); None if L is not 7-smooth."""
    R, cost, m, fac = {2: 4, 4: 16, 8: 52, 3: 14, 5: 36, 7: 66}, 0, L, []
    for r in (8, 4, 2, 3, 5, 7):
        while m % r == 0:
            fac.append(r)
            m //= r
    if m > 1:
        return None
    for i, r in enumerate(fac):
        cost += (L // r) * R[r] + (4 * (L // r) * (r - 1) if i + 1 < len(fac) else 0)
    return cost


def _continuation(n, policy, tab):
    if policy == 0:
        return 27
    ok = [(c, _cost(n + c)) for c in range(27, max(tab) + 1) if _cost(n + c) is not None]
    return min(ok, key=lambda v: (v[1], v[0]))[0] if policy == 2 else ok[0][0]


def exact(case, seed):
    if case["kind"] != "box" or case["op"] not in ("rhs", "noalloc", "filter") or case["n1"] * case["n2"] > 250000:
        return None  # whole steps, other layouts and larger boxes: too long in plain numpy, or no single-pass value
    tab = _tables(5)
    w = workload(case)
    e, mu = _flow(case, w, seed)
    n1, n2 = case["n1"], case["n2"]
    e = e.cpu().numpy().astype(np.longdouble).reshape(4, n2, n1)
    mu = mu.cpu().numpy().astype(np.longdouble).reshape(n2, n1)
    C1, C2 = (_continuation(n, case["policy"], tab) for n in (n1, n2))
    h = np.longdouble(1.0) / (n1 - 1)
    rho, mx, my, E = e
    p = (np.longdouble(GAMMA) - 1) * (E - (mx * mx + my * my) / (2 * rho))
    if case["op"] == "filter":
        def sig(k, L):
            return np.exp(-np.longdouble(10) * np.abs(2 * k / L) ** 14)
        q = np.stack([rho, mx, my, p / rho])
        q = _lines(q, C1, tab, sig)
        q = np.swapaxes(_lines(np.ascontiguousarray(np.swapaxes(q, 1, 2)), C2, tab, sig), 1, 2)
        E = q[0] * q[3] / (np.longdouble(GAMMA) - 1) + (q[1] ** 2 + q[2] ** 2) / (2 * q[0])
        out = np.stack([q[0], q[1], q[2], E])
    else:
        def dif(k, L):
            m = k.copy()
            if L % 2 == 0:
                m[L // 2] = 0
            return 1j * (2 * np.pi * m / (L * h))

        def dx(f):
            return _lines(f, C1, tab, dif)

        def dy(f):
            return np.swapaxes(_lines(np.ascontiguousarray(np.swapaxes(f, 1, 2)), C2, tab, dif), 1, 2)
        u, v = mx / rho, my / rho
        fx = np.stack([mx, mx * u + p, mx * v, u * (E + p)]) - mu * dx(e)
        fy = np.stack([my, my * u, my * v + p, v * (E + p)]) - mu * dy(e)
        out = -(dx(fx) + dy(fy))
    return torch.from_numpy(out.astype(np.float64).reshape(4, n1 * n2))

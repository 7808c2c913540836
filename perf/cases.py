"""Performance cases: the calls a user of this library makes, over the range of sizes they are made at.

listed() names twelve of them; draw(rng) gives further ones of the same ranges.  A case is a dict of plain
values, of one of five kinds:

  grid     time steps (weno_run, weno_ssprk3_step) or the residual (weno_rhs) on a full 1D, 2D or 3D grid
  cross    weno_cross_eval: the pointwise residual on the fibers of a TT-cross sweep
  stage    one stage of a TT time step: weno_tt_round of U + dt L per field, then the residual of the rounded state
           on its fibers
  maxvol   weno_maxvol on the tall matrices a cross sweep selects rows of
  ttcross  weno_tt_cross: a whole fixed-rank cross of the residual

prepare() makes the inputs on the GPU from the seed, run() is one pass, work() its indispensable bytes and
operations, exact() the same values in 64 bits by plain torch.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2405_12301_gb300 import weno as W

GAMMA, EPS, CFL = 1.4, 1e-6, 0.5
BC = {"p": W.BC_PERIODIC, "t": W.BC_TRANSMISSIVE, "r": W.BC_REFLECTIVE}
MODEL = {"euler": W.MODEL_EULER, "advect": W.MODEL_ADVECT, "burgers": W.MODEL_BURGERS}
FOREVER = 1e30


def grid(name=None, dim=2, nx=64, ny=1, nz=1, model="euler", prec="fp64", ic="wave", bc="pp", alpha="global",
         call="run", steps=1):
    c = dict(kind="grid", dim=dim, nx=nx, ny=ny, nz=nz, model=model, prec=prec, ic=ic, bc=bc, alpha=alpha, call=call,
             steps=steps)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the paper's smallest problem: an order study runs thousands of these steps, all of them latency
        grid("run_1d_256_fp64", dim=1, nx=256, call="run", steps=64),
        # the quadrant problem at the size it is validated at, with the conservation sums a run reports
        grid("run_2d_quadrant_256_fp64", dim=2, nx=256, ny=256, ic="quadrant", bc="tt", call="run", steps=4),
        # one step at a time (a user's own loop around weno_ssprk3_step) of the quadrant problem in FP32-bulk
        grid("step_2d_quadrant_1024_bulk", dim=2, nx=1024, ny=1024, prec="bulk", ic="quadrant", bc="tt", call="step"),
        # the largest 2D density wave, as production runs it: graph-replayed steps
        grid("run_2d_wave_2048_bulk", dim=2, nx=2048, ny=2048, prec="bulk", call="run", steps=4),
        # the 3D density wave of the largest memory footprint that a run of this length takes
        grid("run_3d_wave_256_bulk", dim=3, nx=256, ny=256, nz=256, prec="bulk", call="run", steps=2),
        # L(U) in FP64 for a time integrator of the user's own: ragged sizes, walls, a speed per direction
        grid("rhs_3d_ragged_fp64", dim=3, nx=97, ny=83, nz=61, ic="smooth", bc="rt", alpha="dir", call="rhs"),
        # linear advection, the accuracy table's problem
        grid("run_3d_advect_128_fp64", dim=3, nx=128, ny=128, nz=128, model="advect", ic="sine", call="run", steps=1),
        # one cross sweep's fibers of 64 independent instances in one call
        dict(name="cross_64_fp32", kind="cross", count=64, nmin=64, nmax=512, rmin=2, rmax=32, fp64=False, graph=False),
        # one instance, replayed as a graph: a serial solver's inner call
        dict(name="cross_1_graph", kind="cross", count=1, nmin=64, nmax=256, rmin=8, rmax=16, fp64=False, graph=True),
        # one TT-SSPRK3 stage of two instances at full rank
        dict(name="stage_2_rank32", kind="stage", count=2, nmin=64, nmax=256, rmin=24, rmax=32, eps=1e-4),
        # the row selections of one cross step
        dict(name="maxvol_16", kind="maxvol", count=16, nmin=256, nmax=12000, rmin=4, rmax=32),
        # a cross of the residual with 64-bit fibers
        dict(name="ttcross_4_fp64", kind="ttcross", count=4, nmin=48, nmax=128, rmin=4, rmax=10, sweeps=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid"] * 6 + ["cross", "cross", "stage", "maxvol", "ttcross"])
    if kind == "grid":
        dim = rng.choice([1, 2, 2, 2, 3, 3])
        prec = rng.choice(["fp64", "bulk"])
        model = rng.choice(["euler"] * 5 + ["advect", "burgers"]) if prec == "fp64" else "euler"
        if dim == 1:
            n = [_log(rng, 48 if prec == "fp64" else 4096, 200000), 1, 1]
            steps = rng.choice([1, 4, 16, 64]) if n[0] < 4096 else 2
        elif dim == 2:
            lo, hi = (48, 900) if prec == "fp64" else (256, 2000)
            n = [_log(rng, lo, hi), _log(rng, lo, hi), 1]
            steps = rng.choice([1, 2, 4]) if n[0] * n[1] < 300000 else 1
        else:
            lo, hi = (20, 96) if prec == "fp64" else (80, 250)
            n = [_log(rng, lo, hi) for _ in range(3)]
            steps = 1
        call = rng.choice(["run", "run", "step", "rhs"]) if prec == "fp64" else rng.choice(["run", "run", "step"])
        ic = "sine" if model != "euler" else rng.choice(["smooth", "wave", "quadrant"] if dim == 2 else ["smooth", "wave"])
        bc = "pp" if ic == "wave" or model != "euler" else "tt" if ic == "quadrant" else rng.choice(["pp", "tt", "rt", "rr"])
        return grid(dim=dim, nx=n[0], ny=n[1], nz=n[2], model=model, prec=prec, ic=ic, bc=bc,
                    alpha=rng.choice(["global", "global", "dir"]), call=call, steps=steps if call == "run" else 1)
    if kind == "cross":
        r = _log(rng, 3, 32)
        return dict(kind="cross", count=_log(rng, 1, 40), nmin=40, nmax=_log(rng, 64, 500), rmin=max(1, r // 3), rmax=r,
                    fp64=rng.random() < 0.25, graph=rng.random() < 0.3)
    if kind == "stage":
        r = _log(rng, 3, 32)
        return dict(kind="stage", count=_log(rng, 1, 4), nmin=40, nmax=_log(rng, 48, 256), rmin=max(2, r // 2), rmax=r,
                    eps=1e-4)
    if kind == "maxvol":
        r = _log(rng, 3, 48)
        return dict(kind="maxvol", count=_log(rng, 1, 16), nmin=2 * r, nmax=_log(rng, 256, 14000), rmin=max(1, r // 4),
                    rmax=r)
    r = _log(rng, 3, 10)
    return dict(kind="ttcross", count=_log(rng, 1, 6), nmin=32, nmax=_log(rng, 48, 160), rmin=2, rmax=r,
                sweeps=rng.choice([0, 1, 2]))


# ------------------------------------------------------------------ grids
def _dev(x):
    return torch.as_tensor(x, dtype=torch.float64, device="cuda")


def _shape(case):
    return [case["nx"], case["ny"], case["nz"]]


def _length(case):
    return 2.0 if case["ic"] == "wave" else 1.0


def _bcs(case):
    b = (BC[case["bc"][0]], BC[case["bc"][1]])
    return (b, b, b)


def _axes(case, length):
    """Cell-centre coordinates of the three directions, shaped for broadcasting over [nz][ny][nx]."""
    n, out = _shape(case), []
    for d in range(3):
        x = (torch.arange(n[d], dtype=torch.float64, device="cuda") + 0.5) * (length / n[d])
        if d >= case["dim"]:
            x = torch.zeros(1, dtype=torch.float64, device="cuda")
        s = [1, 1, 1]
        s[2 - d] = n[d]
        out.append(x.view(s))
    return out


def _conserved(dim, rho, vel, p):
    ke = sum(v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [p / (GAMMA - 1.0) + 0.5 * rho * ke]).contiguous()


def _initial(case, seed):
    """The seeded initial state [nf][nz][ny][nx]."""
    rng = np.random.default_rng([12301, seed])
    dim, n = case["dim"], _shape(case)
    X, Y, Z = _axes(case, _length(case))
    full = torch.zeros(n[2], n[1], n[0], dtype=torch.float64, device="cuda")
    ph, amp = rng.uniform(0, 2 * np.pi), rng.uniform(0.15, 0.25)
    if case["model"] != "euler":  # offset + sin(2 pi (x + y + z)), the scalar problems' initial state
        return (0.25 + amp * torch.sin(2 * np.pi * (X + Y + Z) + ph) + full)[None].contiguous()
    if case["ic"] == "wave":  # rho = 1 + a sin(pi (x + y + z) + phase), u = v = w = 1, p = 1
        rho = 1.0 + amp * torch.sin(np.pi * (X + Y + Z) + ph) + full
        one = torch.ones_like(full)
        return _conserved(dim, rho, [one] * dim, one)
    if case["ic"] == "quadrant":  # the four states of the quadrant problem, its fronts spread as in a developed run
        sx, sy = rng.uniform(0.45, 0.55, 2)
        wid = 3.0 / max(n[0], n[1])
        E = 0.5 * (1.0 + torch.tanh((X - sx) / wid))
        N = 0.5 * (1.0 + torch.tanh((Y - sy) / wid))
        mix = lambda ne, nw, sw, se: ne * E * N + nw * (1 - E) * N + sw * (1 - E) * (1 - N) + se * E * (1 - N)
        p, rho = mix(1.5, 0.3, 0.029, 0.3), mix(1.5, 0.5323, 0.138, 0.5323)
        return _conserved(2, rho, [mix(0.0, 1.206, 1.206, 0.0), mix(0.0, 0.0, 1.206, 1.206)], p)

    def smooth():  # a random smooth periodic field of size at most 1
        g = full.clone()
        tot = 0.0
        for _ in range(3):
            k, q, a = rng.integers(1, 4, 3), rng.uniform(0, 2 * np.pi, 3), rng.uniform(0.2, 1)
            g += a * torch.sin(2 * np.pi * k[0] * X + q[0]) * torch.sin(2 * np.pi * k[1] * Y + q[1]) \
                * torch.sin(2 * np.pi * k[2] * Z + q[2])
            tot += a
        return g / tot

    rho, p = 1.0 + 0.3 * smooth(), 1.0 + 0.3 * smooth()
    return _conserved(dim, rho, [0.5 * smooth() for _ in range(dim)], p)


def _prepare_grid(case, seed):
    dim, n = case["dim"], _shape(case)
    U = _initial(case, seed)
    s = W.Solver(dim, n[:dim], (0.0,) * dim, (_length(case),) * dim, gamma=GAMMA, eps_weno=EPS, cfl=CFL, bc=_bcs(case),
                 precision=W.FP32_BULK if case["prec"] == "bulk" else W.FP64, model=MODEL[case["model"]],
                 alpha_mode=W.ALPHA_PER_DIR if case["alpha"] == "dir" else W.ALPHA_GLOBAL_NORM)
    s.set_time(0.0)
    st = dict(solver=s, U=U)
    if case["call"] == "rhs":
        st.update(R=torch.empty_like(U), a=torch.empty(1, dtype=torch.float64, device="cuda"))
    return st


def _run_grid(case, st):
    s, U = st["solver"], st["U"]
    if case["call"] == "rhs":
        s.rhs(U, st["R"], st["a"])
        return dict(R=st["R"], alpha=st["a"])
    if case["call"] == "step":
        s.step(U, FOREVER)
        return dict(U=U)
    steps = s.run(U, FOREVER, max_steps=case["steps"], graph_steps=case["steps"])
    out = dict(U=U, steps=int(steps))
    if case["ic"] == "quadrant":
        out["sums"] = np.array(s.sums(U))
    return out


def _exact_grid(case, seed):
    """The scheme in plain torch: WENO5-JS, global or per-direction Lax-Friedrichs splitting, SSP-RK3."""
    dim, n, model = case["dim"], _shape(case), case["model"]
    h = [_length(case) / n[d] for d in range(dim)]
    U = _initial(case, seed)
    nf = U.shape[0]

    def speeds(U):  # (max |u| + a, max |u_d| + a)
        if model == "advect":
            return 1.0, [1.0] * dim
        if model == "burgers":
            a = float(U.abs().max())
            return a, [a] * dim
        v = [U[1 + d] / U[0] for d in range(dim)]
        u2 = sum(x * x for x in v)
        a = (GAMMA * ((GAMMA - 1.0) * (U[-1] - 0.5 * U[0] * u2)) / U[0]).sqrt()
        g = float((u2.sqrt() + a).max())
        return g, [float((x.abs() + a).max()) for x in v] if case["alpha"] == "dir" else [g] * dim

    def flux(U, d):
        if model != "euler":
            return [U[0] if model == "advect" else 0.5 * U[0] * U[0]]
        v = [U[1 + e] / U[0] for e in range(dim)]
        p = (GAMMA - 1.0) * (U[-1] - 0.5 * U[0] * sum(x * x for x in v))
        return [U[1 + d]] + [U[1 + e] * v[d] + (p if e == d else 0.0) for e in range(dim)] + [v[d] * (U[-1] + p)]

    def weno(v0, v1, v2, v3, v4):
        q0, q1, q2 = (2 * v2 + 5 * v3 - v4) / 6, (-v1 + 5 * v2 + 2 * v3) / 6, (2 * v0 - 7 * v1 + 11 * v2) / 6
        b0 = 13 / 12 * (v2 - 2 * v3 + v4) ** 2 + 0.25 * (3 * v2 - 4 * v3 + v4) ** 2
        b1 = 13 / 12 * (v1 - 2 * v2 + v3) ** 2 + 0.25 * (v1 - v3) ** 2
        b2 = 13 / 12 * (v0 - 2 * v1 + v2) ** 2 + 0.25 * (v0 - 4 * v1 + 3 * v2) ** 2
        w0, w1, w2 = 0.3 / (b0 + EPS) ** 2, 0.6 / (b1 + EPS) ** 2, 0.1 / (b2 + EPS) ** 2
        return (w0 * q0 + w1 * q1 + w2 * q2) / (w0 + w1 + w2)

    def rhs(U):
        al = speeds(U)[1]
        R = torch.zeros_like(U)
        for d in range(dim):
            ax, m = 3 - d, n[d]
            src = torch.arange(-3, m + 3, device="cuda")
            ghost = (src < 0) | (src >= m)
            rules = [case["bc"][0] if c < 0 else case["bc"][1] for c in src.tolist()]
            mirror = torch.tensor([r == "r" for r in rules], device="cuda") & ghost
            at = []
            for c, r in zip(src.tolist(), rules):
                if 0 <= c < m:
                    at.append(c)
                elif r == "p":
                    at.append(c % m)
                elif r == "t":
                    at.append(min(max(c, 0), m - 1))
                else:
                    at.append(-1 - c if c < 0 else 2 * m - 1 - c)
            P = U.index_select(ax, torch.tensor(at, device="cuda"))
            if model == "euler":
                s = [1] * 3
                s[ax - 1] = m + 6
                P[1 + d] = torch.where(mirror.view(s), -P[1 + d], P[1 + d])
            F = flux(P, d)
            for f in range(nf):
                fp, fm = 0.5 * (F[f] + al[d] * P[f]), 0.5 * (F[f] - al[d] * P[f])
                cut = lambda v, k: v.narrow(ax - 1, k, m + 1)
                H = weno(*[cut(fp, k) for k in range(5)]) + weno(*[cut(fm, k) for k in range(5, 0, -1)])
                R[f] -= (H.narrow(ax - 1, 1, m) - H.narrow(ax - 1, 0, m)) / h[d]
                del fp, fm, H
        return R

    if case["call"] == "rhs":
        return dict(R=rhs(U), alpha=torch.tensor([speeds(U)[0]], dtype=torch.float64))
    for _ in range(case["steps"]):
        dt = CFL * min(h) / speeds(U)[0]
        U1 = U + dt * rhs(U)
        U2 = 0.75 * U + 0.25 * (U1 + dt * rhs(U1))
        U = U / 3 + 2 / 3 * (U2 + dt * rhs(U2))
    out = dict(U=U, steps=None)
    if case["call"] == "run" and case["ic"] == "quadrant":
        out["sums"] = U.sum(dim=(1, 2, 3)).cpu().numpy()
    return out


def _work_grid(case):
    cells = case["nx"] * case["ny"] * case["nz"]
    dim, euler = case["dim"], case["model"] == "euler"
    nf = dim + 2 if euler else 1
    # per cell and direction: 137 per interface flux and component, 3 per flux difference, the split point fluxes
    res = dim * (nf * 140 + (9 * dim + 18 if euler else 6))
    stages = 0 if case["call"] == "rhs" else 3 * case["steps"]
    flops = cells * (res if case["call"] == "rhs" else stages * (res + 5 * nf + 6 * dim + 10))
    return dict(bytes=2 * 8 * nf * cells, flops=flops)


# ------------------------------------------------------------ TT instances
def _sizes(rng, lo, hi, k):
    return [int(round(math.exp(v))) for v in rng.uniform(math.log(lo), math.log(hi), k)]


def _shapes(case):
    """Modes and ranks of every instance: they belong to the case, the same for each seed."""
    rng = np.random.default_rng([7, case["count"], case["nmax"], case["rmax"]])
    out = []
    for _ in range(case["count"]):
        if case["kind"] == "cross" and case["nmax"] == 512:  # the benchmark's instances: powers of two
            n = [int(rng.choice([64, 128, 256, 512])) for _ in range(3)]
        else:
            n = _sizes(rng, min(case["nmin"], case["nmax"]), case["nmax"], 3)
        out.append((n, [int(v) for v in rng.integers(case["rmin"], case["rmax"] + 1, 2)]))
    return out


def _cores(rng, n, r, mean, size):
    """TT cores (FP64) of mean + size * (a smooth field with a steep front), singular values falling over six decades."""
    x = [(torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) / m for m in n]

    def basis(x, k, m):  # 1, a front four cells wide, then sines and cosines of growing frequency
        freq = torch.arange(k, device="cuda", dtype=torch.float64).view(1, -1) // 2 + 1.0
        B = torch.sin(2 * np.pi * freq * x.view(-1, 1) + _dev(rng.uniform(0, 2 * np.pi, k)).view(1, -1))
        B[:, 0] = 1.0
        if k > 1:
            B[:, 1] = torch.tanh((x - rng.uniform(0.3, 0.7)) / (4.0 / m))
        return B

    A, C = basis(x[0], r[0], n[0]), basis(x[2], r[1], n[2])
    a, b = torch.meshgrid(torch.arange(r[0], device="cuda"), torch.arange(r[1], device="cuda"), indexing="ij")
    decay = 10.0 ** (-6.0 * torch.maximum(a / r[0], b / r[1]) - (a - b).abs().double())
    coef = _dev(rng.uniform(0.3, 1.0, r)) * decay
    coef = coef * (size / coef.sum())
    k = 1.0 + ((a + b) % 3).double()
    M = coef * torch.sin(2 * np.pi * k * x[1].view(-1, 1, 1) + _dev(rng.uniform(0, 2 * np.pi, r)))
    M[:, 0, 0] += mean
    return [A.view(n[0], 1, r[0]).contiguous(), M.contiguous(), C.view(n[2], r[1], 1).contiguous()]


MEANS = (1.0, 0.3, -0.2, 0.25, 2.6)


def _state64(rng, n, r):
    """The five conserved fields of a physical state as FP64 cores."""
    return [_cores(rng, n, r, MEANS[f], 0.15) for f in range(5)]


def _instance(n, r, cores32):
    return dict(n=n, r=r, cores=cores32, h=[1.0 / m for m in n], alpha=2.2,
                bc=[(BC[b], BC[b]) for b in "ptr"])


def _indices(rng, n, r, mode):
    """The left and right multi-indices of a sweep over `mode` (None for an empty side)."""
    draw_ = lambda count, modes: torch.from_numpy(np.stack([rng.integers(0, n[m], count) for m in modes], axis=1)
                                                  .astype(np.int32)).cuda() if modes else None
    return draw_(r[mode - 1] if mode else 1, list(range(mode))), draw_(r[mode] if mode < 2 else 1, list(range(mode + 1, 3)))


def _fibers(rng, shapes, dirs, dtype):
    """Fiber sets of every mode and flux direction, their outputs slices of one buffer."""
    sets, total = [], 0
    for k, (n, r) in enumerate(shapes):
        for fd in dirs:
            for mode in range(3):
                left, right = _indices(rng, n, r, mode)
                size = 5 * (left.shape[0] if mode else 1) * n[mode] * (right.shape[0] if mode < 2 else 1)
                sets.append(dict(instance=k, mode=mode, flux_dir=fd, left=left, right=right, at=total, size=size))
                total += size
    out = torch.zeros(total, dtype=dtype, device="cuda")
    for s in sets:
        s["out"] = out[s["at"]:s["at"] + s["size"]]
    return sets, out


def _rng(case, seed):
    return np.random.default_rng([99, seed])


def _prepare_cross(case, seed):
    rng, shapes = _rng(case, seed), _shapes(case)
    inst = [_instance(n, r, [[c.float() for c in f] for f in _state64(rng, n, r)]) for n, r in shapes]
    sets, out = _fibers(rng, shapes, (0, 1, 2), torch.float64 if case["fp64"] else torch.float32)
    return dict(h=W.weno_init(), inst=inst, sets=sets, out=out)


def _run_cross(case, st):
    W.weno_cross_eval(st["h"], st["inst"], st["sets"], fp64_check=case["fp64"], graph=case["graph"])
    return dict(out=st["out"])


def _mapped(in_, m, c):
    """Index c of mode m after its boundary rule, and where the mirror negates the normal momentum."""
    n = in_["n"][m]
    lo, hi = in_["bc"][m]
    low, high = c < 0, c >= n
    src, flip = c, torch.zeros_like(low)
    for side, rule in ((low, lo), (high, hi)):
        if rule == W.BC_PERIODIC:
            src = torch.where(side, c % n, src)
        elif rule == W.BC_TRANSMISSIVE:
            src = torch.where(side, c.clamp(0, n - 1), src)
        else:
            src = torch.where(side, torch.where(c < 0, -1 - c, 2 * n - 1 - c), src)
            flip = flip | side
    return src, flip


def _point_residual(in_, cores, s):
    """-(F(i+1/2) - F(i-1/2)) / h in direction flux_dir at every sample of a fiber set, FP64, [5][left][n][right]."""
    mode, fd, n = s["mode"], s["flux_dir"], in_["n"]
    li = s["left"].long() if mode else torch.zeros(1, 0, dtype=torch.long, device="cuda")
    ri = s["right"].long() if mode < 2 else torch.zeros(1, 0, dtype=torch.long, device="cuda")
    line = torch.arange(n[mode], device="cuda")

    def value(shift):  # the conserved state at every sample moved by `shift` along fd
        idx, flip = [], None
        for m in range(3):
            c = li[:, m].view(-1, 1, 1) if m < mode else line.view(1, -1, 1) if m == mode else \
                ri[:, m - mode - 1].view(1, 1, -1)
            if m == fd:
                c, flip = _mapped(in_, m, c + shift)
            idx.append(c)
        q = []
        for f in range(5):
            g = [c.double() for c in cores[f]]
            if mode == 0:
                right = torch.einsum("xab,xb->xa", g[1][idx[1].reshape(-1)], g[2][idx[2].reshape(-1), :, 0])
                v = torch.einsum("ia,xa->ix", g[0][idx[0].reshape(-1), 0], right)[None]
            elif mode == 1:
                v = torch.einsum("la,jab,xb->ljx", g[0][idx[0].reshape(-1), 0], g[1][idx[1].reshape(-1)],
                                 g[2][idx[2].reshape(-1), :, 0])
            else:
                left = torch.einsum("la,lab->lb", g[0][idx[0].reshape(-1), 0], g[1][idx[1].reshape(-1)])
                v = torch.einsum("lb,kb->lk", left, g[2][idx[2].reshape(-1), :, 0])[..., None]
            q.append(torch.where(flip, -v, v) if f == 1 + fd else v)
        return q

    fp, fm = [], []
    for k in range(-3, 4):
        q = value(k)
        u = [q[1 + e] / q[0] for e in range(3)]
        p = (GAMMA - 1.0) * (q[4] - 0.5 * q[0] * sum(x * x for x in u))
        F = [q[1 + fd]] + [q[1 + e] * u[fd] + (p if e == fd else 0.0) for e in range(3)] + [u[fd] * (q[4] + p)]
        fp.append([0.5 * (F[f] + in_["alpha"] * q[f]) for f in range(5)])
        fm.append([0.5 * (F[f] - in_["alpha"] * q[f]) for f in range(5)])

    def weno(v):
        b = [13 / 12 * (v[k] - 2 * v[k + 1] + v[k + 2]) ** 2 for k in range(3)]
        b[0] = b[0] + 0.25 * (v[0] - 4 * v[1] + 3 * v[2]) ** 2
        b[1] = b[1] + 0.25 * (v[1] - v[3]) ** 2
        b[2] = b[2] + 0.25 * (3 * v[2] - 4 * v[3] + v[4]) ** 2
        w = [d / (x + EPS) ** 2 for d, x in zip((0.1, 0.6, 0.3), b)]
        c = [(2 * v[0] - 7 * v[1] + 11 * v[2]) / 6, (-v[1] + 5 * v[2] + 2 * v[3]) / 6, (2 * v[2] + 5 * v[3] - v[4]) / 6]
        return sum(x * y for x, y in zip(w, c)) / sum(w)

    out = []
    for f in range(5):
        P, M = [x[f] for x in fp], [x[f] for x in fm]
        lo = weno(P[0:5]) + weno(M[5:0:-1])
        hi = weno(P[1:6]) + weno(M[6:1:-1])
        out.append(-(hi - lo) / in_["h"][fd])
    return torch.stack(out)


def _exact_fibers(inst, cores, sets):
    return torch.cat([_point_residual(inst[s["instance"]], cores[s["instance"]], s).reshape(-1) for s in sets])


def _exact_cross(case, seed):
    st = _prepare_cross(case, seed)
    return dict(out=_exact_fibers(st["inst"], [i["cores"] for i in st["inst"]], st["sets"]))


def _cross_flops(n, r, mode, fd, nl, nr):
    """Per sample: the 7 stencil values of 5 fields, 7 split point fluxes, 2 interfaces, a flux difference; plus the
    contraction of the core rows with the vectors of the side that the stencil does not move."""
    rl, rr = r[mode - 1] if mode else 1, r[mode] if mode < 2 else 1
    length, fixed = (rr, nl) if fd > mode else (rl, nr)
    return nl * n[mode] * nr * (5 * 7 * 2 * length + 7 * 45 + 2 * 5 * 137 + 15) + fixed * 5 * n[mode] * 2 * rl * rr


def _work_cross(case):
    by = fl = 0
    e = 8 if case.get("fp64") else 4
    for n, r in _shapes(case):
        by += 4 * 5 * (n[0] * r[0] + n[1] * r[0] * r[1] + n[2] * r[1])
        for mode in range(3):
            nl, nr = r[mode - 1] if mode else 1, r[mode] if mode < 2 else 1
            fl += sum(_cross_flops(n, r, mode, fd, nl, nr) for fd in range(3))
            by += 3 * 5 * e * nl * n[mode] * nr
    return dict(bytes=by, flops=fl)


# --------------------------------------------------------- TT time stepping
STAGE_DT = 1e-3


def _prepare_stage(case, seed):
    rng, shapes = _rng(case, seed), _shapes(case)
    U = [_state64(rng, n, r) for n, r in shapes]
    L = [[_cores(rng, n, r, 0.0, 1.0) for _ in range(5)] for n, r in shapes]
    sets, out = _fibers(rng, shapes, (0,), torch.float32)
    return dict(h=W.weno_init(), shapes=shapes, U=U, L=L, sets=sets, out=out)


def _run_stage(case, st):
    # F = round(U + dt L) of every field (one batched call), then the residual of F on the next sweep's fibers;
    # the evaluation takes one pair of ranks per instance, so the fields' cores are padded to the largest
    U, L, shapes = st["U"], st["L"], st["shapes"]
    got = W.weno_tt_round(st["h"], [[(1.0, U[k][f]), (STAGE_DT, L[k][f])] for k in range(len(U)) for f in range(5)],
                          case["eps"])
    inst, ranks = [], []
    for k, (n, _) in enumerate(shapes):
        fields = [g for g, _ in got[5 * k:5 * k + 5]]
        r1, r2 = max(c[0].shape[2] for c in fields), max(c[1].shape[2] for c in fields)
        ranks += [c[0].shape[2] for c in fields] + [c[1].shape[2] for c in fields]
        g0 = torch.zeros(5, n[0], 1, r1, device="cuda")
        g1 = torch.zeros(5, n[1], r1, r2, device="cuda")
        g2 = torch.zeros(5, n[2], r2, 1, device="cuda")
        for f, c in enumerate(fields):
            g0[f, :, :, :c[0].shape[2]] = c[0]
            g1[f, :, :c[1].shape[1], :c[1].shape[2]] = c[1]
            g2[f, :, :c[2].shape[1]] = c[2]
        inst.append(_instance(n, [r1, r2], [[g0[f], g1[f], g2[f]] for f in range(5)]))
    W.weno_cross_eval(st["h"], inst, st["sets"])
    return dict(out=st["out"], ranks=np.array(ranks), norms=np.array([v for _, v in got]))


def _exact_stage(case, seed):
    """The rounding as two truncated SVDs of the full tensor's unfoldings."""
    st = _prepare_stage(case, seed)
    inst, cores, norms = [], [], []
    for k, (n, r) in enumerate(st["shapes"]):
        fields = []
        for f in range(5):
            X = sum(c * torch.einsum("ia,jab,kb->ijk", g[0][:, 0], g[1], g[2][:, :, 0])
                    for c, g in ((1.0, st["U"][k][f]), (STAGE_DT, st["L"][k][f])))
            norms.append(float(X.norm()))
            delta = case["eps"] / math.sqrt(2.0) * norms[-1]

            def cut(M):  # (left vectors, S V^T) of the smallest rank whose tail is within delta
                u, s, v = torch.linalg.svd(M, full_matrices=False)
                tail = s.square().flip(0).cumsum(0).sqrt().flip(0)
                q = max(1, int((tail > delta).sum()))
                return u[:, :q], s[:q, None] * v[:q]

            a, rest = cut(X.reshape(n[0], -1))
            b, c = cut(rest.reshape(-1, n[2]))
            fields.append([a.view(n[0], 1, -1), b.view(a.shape[1], n[1], -1).transpose(0, 1).contiguous(),
                           c.t().reshape(n[2], -1, 1)])
        inst.append(_instance(n, None, None))
        cores.append(fields)
    return dict(out=_exact_fibers(inst, cores, st["sets"]), ranks=None, norms=np.array(norms))


def _work_stage(case):
    by, fl = 0, 0
    for n, r in _shapes(case):
        R1, R2 = 2 * r[0], 2 * r[1]
        by += 8 * 5 * 3 * (n[0] * r[0] + n[1] * r[0] * r[1] + n[2] * r[1])
        qr = lambda m, k: 2 * m * k * k - 2 * k ** 3 / 3
        ap = lambda m, k, p: 4 * m * k * p - 2 * k * k * p
        k3, m2 = min(n[2], R2), n[1] * min(n[2], R2)
        k2 = min(m2, R1)
        fl += 5 * (qr(n[2], R2) + qr(m2, R1) + qr(n[0], k2) + qr(r[0] * n[1], k3) + ap(n[0], k2, r[0]) +
                   ap(m2, k2, r[0]) + ap(r[0] * n[1], k3, r[1]) + ap(n[2], k3, r[1]))
        for mode in range(3):
            nl, nr = r[mode - 1] if mode else 1, r[mode] if mode < 2 else 1
            fl += _cross_flops(n, r, mode, 0, nl, nr)
            by += 5 * 4 * nl * n[mode] * nr
    return dict(bytes=by, flops=fl)


# --------------------------------------------------- cross index selection
def _mv_shapes(case):
    rng = np.random.default_rng([5, case["count"], case["nmax"], case["rmax"]])
    out = []
    for _ in range(case["count"]):
        r = int(rng.integers(case["rmin"], case["rmax"] + 1))
        out.append((max(r, _sizes(rng, min(case["nmin"], case["nmax"]), case["nmax"], 1)[0]), r))
    return out


def _prepare_maxvol(case, seed):
    """Fiber matrices: smooth columns of falling size, mixed, as the unfoldings of a cross sweep are."""
    rng, mats = _rng(case, seed), []
    for n, r in _mv_shapes(case):
        x = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n
        B = torch.sin(math.pi * _dev(rng.uniform(0.5, 3.0 * r, r)).view(1, -1) * x.view(-1, 1) +
                      _dev(rng.uniform(0, 2 * np.pi, r)).view(1, -1))
        B = B * 10.0 ** (-3.0 * torch.arange(r, device="cuda", dtype=torch.float64) / r)
        mats.append((B @ _dev(rng.normal(size=(r, r)))).contiguous())
    return dict(h=W.weno_init(), mats=mats)


def _run_maxvol(case, st):
    got = W.weno_maxvol(st["h"], st["mats"])
    return dict(idx=[i for i, _, _ in got], B=[b for _, b, _ in got], swaps=np.array([s for _, _, s in got]))


def _maxvol_rows(A, delta=1e-2, most=200):
    n, r = A.shape
    Wk, chosen, I = A.clone(), torch.zeros(n, dtype=torch.bool, device=A.device), []
    for j in range(r):
        p = int(torch.where(chosen, -1.0, Wk[:, j].abs()).argmax())
        I.append(p)
        chosen[p] = True
        f = torch.where(chosen, 0.0, Wk[:, j] / Wk[p, j])
        Wk -= f[:, None] * Wk[p][None]
    B = torch.linalg.solve(A[I], A, left=False)
    for _ in range(most):
        i, j = divmod(int(B.abs().argmax()), r)
        piv = float(B[i, j])
        if abs(piv) <= 1.0 + delta:
            break
        row = B[i].clone()
        row[j] -= 1.0
        B -= B[:, j:j + 1] * row[None] / piv
        I[j] = i
    return I, torch.linalg.solve(A[I], A, left=False)


def _exact_maxvol(case, seed):
    mats = _prepare_maxvol(case, seed)["mats"]
    return dict(idx=[None] * len(mats), B=[_maxvol_rows(A)[1] for A in mats], swaps=None)


def _work_maxvol(case):
    by = fl = 0
    for n, r in _mv_shapes(case):
        by += 8 * 2 * n * r
        fl += 2 * n * r * r  # the elimination, then B from its multipliers
    return dict(bytes=by, flops=fl)


def _prepare_ttcross(case, seed):
    rng, shapes = _rng(case, seed), _shapes(case)
    inst = [_instance(n, r, [[c.float() for c in f] for f in _state64(rng, n, r)]) for n, r in shapes]
    J1 = [torch.from_numpy(np.stack([rng.integers(0, n[1], r[0]), rng.integers(0, n[2], r[0]),
                                     np.arange(r[0]) % 5], axis=1).astype(np.int32)).cuda() for n, r in shapes]
    J2 = [torch.from_numpy(np.stack([rng.permutation(n[2])[:r[1]], np.arange(r[1]) % 5], axis=1).astype(np.int32)).cuda()
          for n, r in shapes]
    return dict(h=W.weno_init(), inst=inst, ranks=[tuple(r) for _, r in shapes], J1=J1, J2=J2)


def _run_ttcross(case, st):
    # every pass starts from the same index sets, as a solver with its own cross of each stage does
    got = W.weno_tt_cross(st["h"], st["inst"], 0, st["ranks"], [j.clone() for j in st["J1"]],
                          [j.clone() for j in st["J2"]], sweeps=case["sweeps"], fp64_check=True)
    return [dict(cores=g["cores"], I1=g["I1"], I2=g["I2"], J1=g["J1"], J2=g["J2"]) for g in got]


def _exact_ttcross(case, seed):
    st = _prepare_ttcross(case, seed)
    out = []
    for k, in_ in enumerate(st["inst"]):
        n, (r1, r2) = in_["n"], st["ranks"][k]
        J1, J2 = st["J1"][k].long(), st["J2"][k].long()
        at = torch.arange(r1, device="cuda"), torch.arange(r2, device="cuda")

        def fibers(mode, left, right):
            return _point_residual(in_, in_["cores"], dict(mode=mode, flux_dir=0, left=left, right=right))

        for it in range(case["sweeps"] + 1):
            F0 = fibers(0, None, J1[:, :2])
            I1, B1 = _maxvol_rows(F0[J1[:, 2], 0, :, at[0]].t().contiguous())
            I1 = torch.tensor(I1, device="cuda")
            F1 = fibers(1, I1[:, None], J2[:, :1])
            sel, B2 = _maxvol_rows(F1[J2[:, 1], :, :, at[1]].permute(1, 2, 0).reshape(r1 * n[1], r2).contiguous())
            sel = torch.tensor(sel, device="cuda")
            I2 = torch.stack([I1[sel // n[1]], sel % n[1]], dim=1)
            F2 = fibers(2, I2, None)[..., 0]  # [5][r2][n3]
            if it == case["sweeps"]:
                break
            sel = torch.tensor(_maxvol_rows(F2.permute(2, 0, 1).reshape(-1, r2).contiguous())[0], device="cuda")
            J2 = torch.stack([sel // 5, sel % 5], dim=1)
            F1 = fibers(1, I1[:, None], J2[:, :1])
            R1 = F1[J2[:, 1], :, :, at[1]].permute(2, 0, 1).reshape(n[1] * r2, r1).contiguous()  # rows (j, b)
            sel = torch.tensor(_maxvol_rows(R1)[0], device="cuda")
            J1 = torch.cat([(sel // r2)[:, None], J2[sel % r2]], dim=1)
        out.append(dict(cores=[B1.view(n[0], 1, r1), B2.view(r1, n[1], r2).transpose(0, 1).contiguous(),
                               F2.permute(2, 1, 0).contiguous()], I1=None, I2=None, J1=None, J2=None))
    return out


def _work_ttcross(case):
    by = fl = 0
    for n, r in _shapes(case):
        by += 4 * 5 * (n[0] * r[0] + n[1] * r[0] * r[1] + n[2] * r[1]) + 8 * (n[0] * r[0] + n[1] * r[0] * r[1] + 5 * n[2] * r[1])
        for mode, times in ((0, case["sweeps"] + 1), (1, 2 * case["sweeps"] + 1), (2, case["sweeps"] + 1)):
            nl, nr = r[mode - 1] if mode else 1, r[mode] if mode < 2 else 1
            fl += times * (_cross_flops(n, r, mode, 0, nl, nr) + 2 * nl * n[mode] * nr * max(r))
    return dict(bytes=by, flops=fl)


# ------------------------------------------------------------------- entry
class _Handle:
    """Frees a handle when its state goes away."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        try:
            W.weno_destroy(self.h)
        except Exception:
            pass


def _of(case, what):
    return globals()["_%s_%s" % (what, case["kind"])]


def prepare(case, seed):
    st = _of(case, "prepare")(case, seed)
    if isinstance(st.get("h"), ctypes.c_void_p):
        st["owner"] = _Handle(st["h"])
    st["case"] = case
    return st


def run(state):
    return _of(state["case"], "run")(state["case"], state)


def work(case):
    return _of(case, "work")(case)


def exact(case, seed):
    if case["kind"] == "stage" and case["nmax"] > 256:
        return None
    return _of(case, "exact")(case, seed)

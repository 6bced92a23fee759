"""The work that users of this framework give it, as cases to be measured.

A case is a dict of plain values.  listed() gives the named cases, draw(rng) one
more of the same ranges, prepare(case, seed) what a program holds before the
call (its inputs on the GPU and the grid, batch or server it keeps), run(state)
one pass through the public entry points of paper_2208_14703_gb300.m1, work(case)
what the pass cannot do without, and exact(case, seed) the pass's outputs from
plain torch in 64 bits where that is quick.

A step's pass sets the state v^n on the device, takes one implicit step and
reads v^{n+1} on the device: what a radiation-hydrodynamics program does once per
time step, its gas update having changed the state in between.  The opacities
and the walls are set once, as they are for such a program's frozen opacities.
The strip shapes are the table that ships beside the package (m1.set_tuning),
which spares a program the tuning launches.

Problems (those of the package's own inputs, benchmark and tests, drawn on the
GPU from the seed): lognormal opacities log10 sigma = 1 + 3 g clipped to [-2, 4],
g a Gaussian random field of correlation length 8 cells;
  gauss  1D, sigma = 1, E = 1e-2 + a Gaussian pulse, periodic, CFL 50
  bump   1D or 2D Gaussian pulse on lognormal opacities (1D periodic, CFL 50;
         2D reflecting walls, CFL 100)
  hot    T = 1 with a hot box at T = 4, E = T^4, reflecting walls, CFL 100
  mixed  the hot box with walls periodic in x, Neumann and reflecting in y
  beam   an f = 1 beam entering the low x wall into a thin channel through the
         lognormal medium, CFL 100
  paper  the paper's own beam: no matter, f = 1 at 45 degrees, CFL 2000, tol 1e-2
  random random admissible states and lognormal opacities (single sweeps)
"""
import json
import math
import os

import torch

from paper_2208_14703_gb300 import m1

# The strip shapes shipped with the package, installed once per process.
_TABLE = os.path.join(os.path.dirname(os.path.abspath(m1.__file__)), "tune_gb300.json")
if os.path.exists(_TABLE):
    with open(_TABLE) as _fh:
        m1.set_tuning(json.load(_fh))

DEV = "cuda"
CYCLES = {"v": 0, "w": 1, "f": 2}


def _step(name, problem, nx, ny, nz, lmax, precision="fp64", cycle="v", tol=1e-8, rule="abs"):
    return dict(name=name, kind="step", problem=problem, nx=nx, ny=ny, nz=nz, lmax=lmax,
                precision=precision, cycle=cycle, tol=tol, rule=rule)


def listed():
    return [
        # the smallest simulation: a 1D pulse, a few hundred cells, all latency
        _step("pulse 1D 256", "gauss", 256, 1, 1, 4, tol=1e-10),
        # a small 2D simulation with ragged sides and mixed walls
        _step("hot 2D 320x208", "mixed", 320, 208, 1, 5),
        # the plain-FP64 workload of the benchmark
        _step("hot 2D 1024 fp64", "hot", 1024, 1024, 1, 8),
        # the same step in mixed precision, the ordinary production choice
        _step("hot 2D 1024 mixed", "hot", 1024, 1024, 1, 8, precision="mixed"),
        # the mixed-precision configuration (a beam in a channel) at a large size
        _step("beam 2D 3072 mixed", "beam", 3072, 3072, 1, 10, precision="mixed"),
        # the paper's own beam, on the cycle shape that suits it
        _step("paper beam 512 W", "paper", 512, 512, 1, 4, cycle="w", tol=1e-2),
        # many independent simulations stepped together (the batched configuration's
        # sizes), mixed precision
        dict(name="batch of 24 mixed", kind="batch", problem="bump", count=24, lo=64, hi=512, lmax=5,
             precision="mixed", cycle="v", tol=1e-8, rule="abs"),
        # a small batch in FP64, 1D and 2D together
        dict(name="batch of 10 fp64", kind="batch", problem="bump", count=10, lo=64, hi=192, lmax=5,
             precision="fp64", cycle="v", tol=1e-8, rule="signed"),
        # requests of several steps served as they come, both lanes
        dict(name="serve 8 mixed", kind="serve", problem="bump", count=8, lo=128, hi=384, lmax=5,
             precision="mixed", cycle="v", tol=1e-8, rule="signed", steps=3),
        # a 3D step
        _step("hot 3D 64", "hot", 64, 64, 64, 4),
        # the paper's first algorithm alone (its Table 1): 20 Jacobi sweeps, FP64
        dict(name="jacobi 2D 2048 fp64", kind="jacobi", problem="random", nx=2048, ny=2048, nz=1,
             precision="fp64", sweeps=20),
        # the 3D operator alone on a grid far over L2
        dict(name="jacobi 3D 192", kind="jacobi", problem="random", nx=192, ny=192, nz=192,
             precision="fp64", sweeps=4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, lo, hi, lmax):
    d = 1 << (lmax - 1)
    return max(2, round(_log(rng, lo, hi) / d)) * d


def draw(rng):
    kind = rng.choice(["1d", "1d", "2d", "2d", "2d", "2d", "beam", "paper", "batch", "serve", "3d",
                       "3d", "j2", "j3"])
    prec = rng.choice(["fp64", "mixed"])
    cyc = rng.choice(["v", "v", "v", "f", "w"])
    if kind == "1d":
        lmax = rng.randint(3, 6)
        n = _size(rng, 128, 65536, lmax)
        return dict(_step("", rng.choice(["gauss", "bump"]), n, 1, 1, lmax, prec, "v", 1e-8,
                          "signed"), name="1d")
    if kind == "2d":
        lmax = rng.randint(3, 7)
        nx = _size(rng, 48, 700 if prec == "fp64" else 1400, lmax)
        ny = _size(rng, nx / 2, min(nx * 2, 1500), lmax)
        return dict(_step("", rng.choice(["hot", "mixed"]), nx, ny, 1, lmax, prec,
                          cyc if lmax < 6 else "v", 1e-8, "abs"), name="2d")
    if kind == "beam":
        lmax = rng.randint(5, 8)
        n = _size(rng, 128, 512 if prec == "fp64" else 1536, lmax)
        return dict(_step("", "beam", n, n, 1, lmax, prec, "v", 1e-8, "abs"), name="beam")
    if kind == "paper":
        lmax = rng.randint(1, 4)
        n = _size(rng, 64, 512, lmax)
        return dict(_step("", "paper", n, n, 1, lmax, "fp64", rng.choice(["v", "w", "f"]), 1e-2),
                    name="paper")
    if kind == "batch":
        hi = 16 * round(_log(rng, 96, 320) / 16)
        return dict(name="batch", kind="batch", problem="bump", count=rng.randint(2, 16), lo=64,
                    hi=hi, lmax=5, precision=prec, cycle="v", tol=1e-8, rule="signed")
    if kind == "serve":
        return dict(name="serve", kind="serve", problem="bump", count=rng.randint(2, 6), lo=64,
                    hi=16 * rng.randint(8, 20), lmax=5, precision=prec, cycle="v", tol=1e-8,
                    rule="signed", steps=rng.randint(1, 3))
    if kind == "3d":
        lmax = rng.randint(2, 4)
        nx, ny, nz = (_size(rng, 16, 72, lmax) for _ in range(3))
        return dict(_step("", rng.choice(["hot", "mixed", "beam"]), nx, ny, nz, lmax, "fp64",
                          cyc, 1e-8, "abs"), name="3d")
    if kind == "j2":
        nx = round(_log(rng, 30, 2048))
        return dict(name="j2", kind="jacobi", problem="random", nx=nx,
                    ny=round(_log(rng, 30, 2048)), nz=1, precision="fp64", sweeps=rng.randint(1, 20))
    return dict(name="j3", kind="jacobi", problem="random", nx=round(_log(rng, 12, 192)),
                ny=round(_log(rng, 12, 192)), nz=round(_log(rng, 12, 192)), precision="fp64",
                sweeps=rng.randint(1, 4))


# ---- inputs ---------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)


def _opacity(shape, g, corr=8.0):
    """log10 sigma = 1 + 3 g clipped to [-2, 4], g a unit Gaussian random field."""
    x = torch.fft.fftn(torch.randn(shape, generator=g, device=DEV, dtype=torch.float64))
    k2 = 0.0
    for a, n in enumerate(shape):
        f = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64) ** 2
        k2 = k2 + f.reshape([-1 if b == a else 1 for b in range(len(shape))])
    x = torch.fft.ifftn(x * torch.exp(-0.5 * (2 * math.pi * corr) ** 2 * k2)).real
    x = x - x.mean()
    x = x / x.std(unbiased=False).clamp_min(1e-30)
    return 10.0 ** torch.clamp(1.0 + 3.0 * x, -2.0, 4.0)


def _centres(n, h, lo=0.0):
    return lo + (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) * h


def _grid_shape(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    return (nz, ny, nx) if nz > 1 else (ny, nx) if ny > 1 else (nx,)


def _problem(case, seed):
    """shape, h, dt, walls (per axis x, y, z: low, high), state planes (E, F..., T),
    opacities (sa, ss) and the inflow fields on the low x wall (or None)."""
    g = _gen(seed)
    shape = _grid_shape(case)
    d, p = len(shape), case["problem"]
    h = (2.0 if p == "paper" else 1.0) / case["nx"]
    walls = [["reflect", "reflect"] for _ in range(d)]
    T = torch.ones(shape, device=DEV, dtype=torch.float64)
    F = torch.zeros((d,) + shape, device=DEV, dtype=torch.float64)
    inflow, cfl = None, 100.0
    if p in ("gauss", "bump"):
        u = _rand(g, 4).tolist()
        amp = 1.0 + 0.5 * u[0] if p == "gauss" else 1.0 + 99.0 * u[0]
        w = 0.005 if p == "gauss" else 0.002 + 0.018 * u[3]
        r2 = 0.0
        for a in range(d):
            x = _centres(shape[d - 1 - a], h) - (0.25 + 0.5 * u[1 + min(a, 1)])
            r2 = r2 + (x ** 2).reshape([-1 if b == d - 1 - a else 1 for b in range(d)])
        E = 1e-2 + amp * torch.exp(-r2 / w) + torch.zeros_like(T)
        if d == 1:
            walls, cfl = [["periodic", "periodic"]], 50.0
        sa = torch.ones_like(T) if p == "gauss" else _opacity(shape, g)
        ss = torch.ones_like(T) if p == "gauss" else _opacity(shape, g)
    elif p in ("hot", "mixed"):
        box = torch.ones(shape, device=DEV, dtype=torch.bool)
        for a in range(d):
            n = shape[a]
            x = (torch.arange(n, device=DEV) + 0.5) / n
            box &= ((x - 0.5).abs() < 1 / 16).reshape([-1 if b == a else 1 for b in range(d)])
        T = torch.where(box, 4.0, 1.0).to(torch.float64)
        E = T ** 4
        sa, ss = _opacity(shape, g), _opacity(shape, g)
        if p == "mixed":
            walls[0] = ["periodic", "periodic"]
            walls[1] = ["neumann", "reflect"]
    elif p == "beam":
        E = torch.ones_like(T)
        sa, ss = _opacity(shape, g), _opacity(shape, g)
        chan = torch.ones(shape[:-1] if d > 1 else (1,), device=DEV, dtype=torch.bool)
        for a in range(d - 1):
            x = (torch.arange(shape[a], device=DEV) + 0.5) / shape[a]
            chan &= ((x - 0.5).abs() <= (0.05 if d == 2 else 1 / 16)).reshape(
                [-1 if b == a else 1 for b in range(d - 1)])
        sa[chan], ss[chan] = 1e-2, 1e-2
        walls[0][0] = "inflow"
        inflow = [torch.ones(chan.shape, dtype=torch.float64), chan.to(torch.float64).cpu()]
        inflow += [torch.zeros(chan.shape, dtype=torch.float64)] * (d - 1)
    elif p == "paper":
        E = torch.ones_like(T)
        sa, ss = torch.zeros_like(T), torch.zeros_like(T)
        u = _rand(g, 2).tolist()
        y = _centres(case["ny"], h, -1.0).cpu()
        beam = (y >= -0.875 + 0.1 * u[0]) & (y <= -0.75 + 0.1 * u[0])
        eb = ((1000.0 + 50.0 * u[1]) / 300.0) ** 4
        one, zero = torch.ones_like(y), torch.zeros_like(y)
        inflow = [torch.where(beam, eb * one, one)] + [torch.where(beam, eb / math.sqrt(2.0) * one, zero)] * 2
        walls = [["inflow", "neumann"], ["neumann", "neumann"]]
        cfl = 2000.0
    else:
        E = 10.0 ** (2.0 * _rand(g, *shape) - 1.0)
        F = torch.randn((d,) + shape, generator=g, device=DEV, dtype=torch.float64)
        F = 0.95 * _rand(g, *shape) * E * F / F.norm(dim=0)
        T = 10.0 ** (0.6 * _rand(g, *shape) - 0.3)
        sa, ss = _opacity(shape, g), _opacity(shape, g)
        cfl = 20.0
    state = torch.cat([E[None], F, T[None]]).contiguous()
    return dict(shape=shape, h=h, dt=cfl * h, walls=walls, state=state,
                sig=torch.stack([sa, ss]).contiguous(), inflow=inflow)


def _params(case):
    return m1.m1_default_params(tol=case["tol"], max_cycles=1500, cycle=CYCLES[case["cycle"]],
                                dtau_rule=m1.DTAU_SIGNED if case["rule"] == "signed" else m1.DTAU_ABS)


def _desc2(pb, lmax, precision):
    shape, h = pb["shape"], pb["h"]
    nx, ny = shape[-1], shape[0] if len(shape) == 2 else 1
    bc = [w for pair in pb["walls"] for w in pair] + ["periodic"] * (4 - 2 * len(pb["walls"]))
    return m1.make_desc(len(shape), nx, ny, nx * h, ny * h if len(shape) == 2 else 1.0, bc, lmax,
                        precision=m1.MIXED if precision == "mixed" else m1.FP64)


def _planes2(pb):
    """(E, Fx, Fy, T) device tensors of a 1D or 2D problem."""
    s = pb["state"]
    if len(pb["shape"]) == 1:
        return [s[0], s[1], torch.zeros_like(s[0]), s[2]]
    return [s[0], s[1], s[2], s[3]]


def _grid2(pb, lmax, precision):
    grid = m1.Grid(_desc2(pb, lmax, precision))
    planes = _planes2(pb)
    torch.cuda.synchronize()
    grid.set_state(*planes, pb["sig"][0], pb["sig"][1], on_device=True)
    if pb["inflow"] is not None:
        grid.set_inflow(0, *[f.numpy() for f in pb["inflow"]])
    return grid, planes


def _bump_sizes(case, seed):
    """Sizes of a batch's or a server's simulations: by their rank over the whole
    range (the smallest and the largest always there), every fourth one 1D."""
    out = []
    for k in range(case["count"]):
        t = k / max(1, case["count"] - 1)
        n = 16 * round(case["lo"] * (case["hi"] / case["lo"]) ** t / 16)
        out.append((n * 16, 1) if k % 4 == 1 else (n, n))
    return out


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, kind=kind)
    if kind == "step" and case["nz"] > 1:
        pb = _problem(case, seed)
        nz, ny, nx = pb["shape"]
        h = pb["h"]
        bc = tuple(w for pair in pb["walls"] for w in pair)
        grid = m1.Grid3(m1.make_desc3(nx, ny, nz, nx * h, ny * h, nz * h, bc), case["lmax"])
        torch.cuda.synchronize()
        if pb["inflow"] is not None:
            face = torch.zeros(6, 4, max(ny * nz, nx * nz, nx * ny), dtype=torch.float64)
            for f in range(4):
                face[0, f, :ny * nz] = pb["inflow"][f].reshape(-1)
            grid.set_inflow(face.numpy())
        st.update(grid=grid, state=pb["state"], sig=pb["sig"], dt=pb["dt"], params=_params(case),
                  out=torch.empty_like(pb["state"]))
    elif kind == "step":
        pb = _problem(case, seed)
        grid, planes = _grid2(pb, case["lmax"], case["precision"])
        st.update(grid=grid, planes=planes, dt=pb["dt"], params=_params(case),
                  out=[torch.empty_like(x) for x in planes])
    elif kind in ("batch", "serve"):
        pbs = [_problem(dict(problem="bump", nx=nx, ny=ny, nz=1), seed * 64 + k)
               for k, (nx, ny) in enumerate(_bump_sizes(case, seed))]
        st.update(dts=[pb["dt"] for pb in pbs], params=_params(case),
                  planes=[_planes2(pb) for pb in pbs])
        torch.cuda.synchronize()
        if kind == "batch":
            b = m1.Batch([_desc2(pb, case["lmax"], case["precision"]) for pb in pbs])
            for k, pb in enumerate(pbs):
                b.set_state(k, *st["planes"][k], pb["sig"][0], pb["sig"][1], on_device=True)
            st["batch"] = b
        else:
            st["grids"] = [_grid2(pb, case["lmax"], case["precision"])[0] for pb in pbs]
            st["out"] = [[torch.empty_like(x) for x in p] for p in st["planes"]]
            st["server"] = m1.Server(16 << 30, case["count"], case["lmax"],
                                     m1.MIXED if case["precision"] == "mixed" else m1.FP64)
    else:
        pb = _problem(case, seed)
        # the right-hand side of Algorithm 1 in 3D is the caller's
        st.update(dt=pb["dt"], sweeps=case["sweeps"])
        if case["nz"] > 1:
            nz, ny, nx = pb["shape"]
            h = pb["h"]
            st.update(desc=m1.make_desc3(nx, ny, nz, nx * h, ny * h, nz * h, ("reflect",) * 6),
                      state=pb["state"], sig=pb["sig"], rhs=pb["state"].clone(),
                      out=torch.empty_like(pb["state"]))
        else:
            grid, planes = _grid2(pb, 1, case["precision"])
            st.update(grid=grid, planes=planes, out=[torch.empty_like(x) for x in planes])
    torch.cuda.synchronize()
    return st


def run(st):
    kind = st["kind"]
    if kind == "step" and "state" in st:
        g = st["grid"]
        g.set_state(st["state"], st["sig"], on_device=True)
        g.implicit_step(st["dt"], st["params"], allow_not_converged=True)
        return g.get_state(st["out"], on_device=True)
    if kind == "step":
        g = st["grid"]
        g.set_state(*st["planes"], on_device=True)
        g.implicit_step(st["dt"], st["params"], allow_not_converged=True)
        return g.get_state(st["out"], on_device=True)
    if kind == "batch":
        b = st["batch"]
        for k, p in enumerate(st["planes"]):
            b.set_state(k, *p, on_device=True)
        b.implicit_step(st["dts"], st["params"], allow_not_converged=True)
        # one flat array per simulation: E, Fx, Fy, T
        return [torch.cat([torch.from_numpy(x).reshape(-1) for x in b.get_state(k)])
                for k in range(len(b))]
    if kind == "serve":
        srv, tickets = st["server"], []
        for k, g in enumerate(st["grids"]):
            g.set_state(*st["planes"][k], on_device=True)
            tickets.append(srv.submit(g, st["case"]["steps"], st["dts"][k], st["params"]))
        for t in tickets:
            srv.wait(t)
        return [g.get_state(o, on_device=True) for g, o in zip(st["grids"], st["out"])]
    if "grid" in st:
        g = st["grid"]
        g.set_state(*st["planes"], on_device=True)
        g.jacobi(st["dt"], st["sweeps"])
        return g.get_state(st["out"], on_device=True)
    out, _ = m1.m1_op_level3(st["desc"], st["dt"], st["sig"], st["state"], rhs=st["rhs"],
                             mode=m1.OP3_JACOBI, sweeps=st["sweeps"], out=st["out"], on_device=True)
    return out


# ---- what a pass cannot do without ------------------------------------------------
# Cycles of a step: what the workloads take to their tolerance (the method's count,
# not the code's).  A cell-update's arithmetic: closure, neighbour terms, right-hand
# side and local solve, one operation per multiply, add or fused pair, in two flops.
_NOMINAL = {"gauss": 150, "bump": 300, "hot": 450, "mixed": 450, "beam": 370, "paper": 30}


def work(case):
    if case["kind"] in ("batch", "serve"):
        total = {"bytes": 0.0, "flops": 0.0}
        for nx, ny in _bump_sizes(case, 0):
            w = work(dict(kind="step", problem="bump", nx=nx, ny=ny, nz=1, sweeps=1))
            for k in total:
                total[k] += w[k] * case.get("steps", 1)
        return total
    n = case["nx"] * case["ny"] * case["nz"]
    d = len(_grid_shape(case))
    ops = {1: 60, 2: 103, 3: 139}[d]
    fields = 5 if d == 3 else 4
    if case["kind"] == "jacobi":
        extra = fields if d == 3 else 0                       # 3D: the right-hand side is read too
        return {"bytes": 8.0 * n * (2 * fields + 2 + extra), "flops": 2.0 * ops * n * case["sweeps"]}
    # six fine sweeps a cycle; the coarse levels add their share of cells
    sweeps = _NOMINAL[case["problem"]] * 6 * (1.0 + 1.0 / (2 ** d - 1))
    return {"bytes": 8.0 * n * (2 * fields + 2), "flops": 2.0 * ops * n * sweeps}


# ---- plain torch in 64 bits -------------------------------------------------------
def _pressure(E, F):
    """The M1 pressure tensor P[a][b] (c = 1)."""
    d = F.shape[0]
    f2 = ((F / E) ** 2).sum(0).clamp(max=1.0)
    s = torch.sqrt(4.0 - 3.0 * f2)
    iso, q = (s - 1.0) / 3.0 * E, 3.0 / (2.0 + s) / E
    return [[q * F[a] * F[b] + (iso if a == b else 0.0) for b in range(d)] for a in range(d)]


def _ghosted(x, axis, low, high, sign):
    """x with one ghost layer on `axis`: wrap, mirror (times `sign`) or copy."""
    n = x.shape[axis]
    first, last = x.narrow(axis, 0, 1), x.narrow(axis, n - 1, 1)
    a = last if low == "periodic" else first * (sign if low == "reflect" else 1.0)
    b = first if high == "periodic" else last * (sign if high == "reflect" else 1.0)
    return torch.cat([a, x, b], axis)


def _neighbours(E, F, pb):
    """The neighbour terms of the Rusanov faces (c = 1): (N_E, N_F[...])."""
    d, dt, h = F.shape[0], pb["dt"], pb["h"]
    beta = dt / (2.0 * h)
    P = _pressure(E, F)
    NE, NF = torch.zeros_like(E), [torch.zeros_like(E) for _ in range(d)]
    for a in range(d):                     # axis a = x, y, z is tensor dimension d - 1 - a
        ax = d - 1 - a
        low, high = pb["walls"][a]
        n = E.shape[ax]

        def pair(x, sign=1.0):
            g = _ghosted(x, ax, low, high, sign)
            return g.narrow(ax, 0, n), g.narrow(ax, 2, n)
        w, e = pair(E)
        fw, fe = pair(F[a], -1.0)
        NE = NE + beta * ((w + e) + (fw - fe))
        for b in range(d):
            gw, ge = pair(F[b], -1.0 if b == a else 1.0)
            pw, pe = pair(P[a][b], 1.0 if b == a else -1.0)
            NF[b] = NF[b] + beta * ((gw + ge) + (pw - pe))
    return NE, torch.stack(NF)


def _solve_gas(C, K, R):
    """The root of C T + K T^4 = R by Newton from the right."""
    T = torch.minimum(R / C, torch.where(K > 0, (R / K.clamp_min(1e-300)) ** 0.25, R / C))
    for _ in range(60):
        T = T - (C * T + K * T ** 4 - R) / (C + 4.0 * K * T ** 3)
    return T


def _jacobi(pb, sweeps):
    d = len(pb["shape"])
    dt, h = pb["dt"], pb["h"]
    E, F, T = pb["state"][0], pb["state"][1:1 + d], pb["state"][1 + d]
    bE, bF, bT = E, F, T
    A = 1.0 + d * dt / h
    ka, kt = dt * pb["sig"][0], dt * (pb["sig"][0] + pb["sig"][1])
    kk = ka / (A + ka)
    for _ in range(sweeps):
        NE, NF = _neighbours(E, F, pb)
        rE = bE + NE
        F = (bF + NF) / (A + kt)
        T = _solve_gas(1.0, A * kk, bT + kk * rE)
        E = (rE + ka * T ** 4) / (A + ka)
    return torch.cat([E[None], F, T[None]])


def _newton_1d(pb):
    """The implicit step's solution on a small periodic 1D grid: dense Newton."""
    n, dt, h = pb["shape"][0], pb["dt"], pb["h"]
    A = 1.0 + dt / h
    ka, kt = dt * pb["sig"][0], dt * (pb["sig"][0] + pb["sig"][1])
    b = torch.cat([pb["state"][0], pb["state"][1], pb["state"][2]])

    def residual(u):
        E, F, T = u[:n], u[n:2 * n], u[2 * n:]
        NE, NF = _neighbours(E, F[None], pb)
        src = ka * (E - T ** 4)
        return torch.cat([A * E + src - NE, (A + kt) * F - NF[0], T - src]) - b
    v = _jacobi(pb, 200).reshape(-1)
    for _ in range(40):
        r = residual(v)
        step = torch.linalg.solve(torch.func.jacrev(residual)(v), r)
        t = 1.0
        while t > 1e-6 and residual(v - t * step).norm() > r.norm():
            t *= 0.5
        v = v - t * step
        if step.norm() <= 1e-14 * v.norm():
            break
    return v.reshape(3, n)


def exact(case, seed):
    if case["kind"] == "jacobi":
        pb = _problem(case, seed)
        s = _jacobi(pb, case["sweeps"])
        return s if case["nz"] > 1 else [s[k] for k in range(4)]
    if case["kind"] == "step" and case["problem"] == "gauss" and case["nx"] <= 512:
        pb = _problem(case, seed)
        s = _newton_1d(pb)
        return [s[0], s[1], torch.zeros_like(s[0]), s[2]]
    return None                            # a converged step is no quick sum in plain torch

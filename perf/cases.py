"""Timed workloads of the solver, each through the entry points a program calls.

A case names a flow (`flow`), its grid, the precision and what is called (`call`):

  step      Solver.step(U, nsteps) from a given state (CFL time step), as a time-marching program does
  rhs       Solver.rhs(U), as a program with its own time integrator does
  adjoint   Solver.adjoint_step with the step's stored stage states: one link of a gradient's
            backward sweep
  serve     a serve.Server given several solves of uneven sizes at once, until their states are back

`prepare` makes what the program holds before the call: the solver (or server) and seeded states on
the GPU.  `exact` is the same arithmetic in plain 64-bit torch, with automatic differentiation for
the adjoint; it shares no code with the solver.
"""
import math
from fractions import Fraction

import numpy as np
import torch

from paper_2406_19494_gb300 import workloads as wl

H = 3                      # halo cells per side of an active axis


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: the 1-D shock tube every solver is tried on first, twenty steps
        dict(name="sod 200", flow="sod", nx=200, ny=1, nz=1, call="step", nsteps=20, precision="fp64"),
        # the smallest 2-D solve of a parameter sweep (inviscid, periodic)
        dict(name="vortex 64x64", flow="vortex", nx=64, ny=64, nz=1, call="step", nsteps=10,
             precision="fp64"),
        # the largest 2-D solve of the serving range: shocks and contacts, transmissive ends
        dict(name="riemann 1024x1024", flow="riemann", nx=1024, ny=1024, nz=1, call="step", nsteps=1,
             precision="fp64"),
        # supersonic laminar boundary layer at its published resolution: inflow, adiabatic wall,
        # stretched grid, Sutherland's law
        dict(name="boundary layer 300x200", flow="layer", nx=300, ny=200, nz=1, call="step", nsteps=5,
             precision="fp64"),
        # a ragged box with walls, WENO5-JS and constant viscosity, one right-hand side for a
        # program that integrates in time by itself
        dict(name="box 61x47x53 rhs", flow="box", nx=61, ny=47, nz=53, call="rhs", nsteps=1,
             precision="fp64"),
        # the headline workload: Taylor-Green vortex at 128^3
        dict(name="tgv 128", flow="tgv", nx=128, ny=128, nz=128, call="step", nsteps=1,
             precision="fp64"),
        # the turbulent channel with its own scheme (TENO6-A, sixth-order dissipative fluxes)
        dict(name="channel 192x128x128", flow="channel", nx=192, ny=128, nz=128, call="step", nsteps=1,
             precision="fp64"),
        # backward sweep of the porous-wall optimisation
        dict(name="porous layer 512x128 adjoint", flow="porous", nx=512, ny=128, nz=1, call="adjoint",
             nsteps=1, precision="fp64"),
        # the mixed-precision path: the smallest 3-D solve of the serving range, the headline
        # size, and a production-size grid
        dict(name="tgv 32 mixed", flow="tgv", nx=32, ny=32, nz=32, call="step", nsteps=10,
             precision="mixed"),
        dict(name="tgv 128 mixed", flow="tgv", nx=128, ny=128, nz=128, call="step", nsteps=2,
             precision="mixed"),
        dict(name="tgv 256 mixed", flow="tgv", nx=256, ny=256, nz=256, call="step", nsteps=1,
             precision="mixed"),
        # eight requests of uneven sizes through the request loop (vortices, Riemann problems,
        # Taylor-Green vortices)
        dict(name="serve 8 solves", flow="sweep", nx=160, ny=160, nz=40, call="serve", nsteps=10,
             precision="fp64"),
    ]


def draw(rng):
    """One more case: sizes log-uniform over the range of its flow, odd ones among them."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    flow = rng.choice(["sod", "vortex", "riemann", "layer", "box", "tgv", "tgv", "tgv mixed", "tgv mixed",
                       "channel", "porous", "vortex mixed", "sweep"])
    if flow == "sod":
        return dict(flow="sod", nx=size(50, 20000), ny=1, nz=1, call="step", nsteps=rng.randint(5, 20),
                    precision="fp64")
    if flow in ("vortex", "riemann", "vortex mixed"):
        n = size(48, 1024)
        return dict(flow=flow.split()[0], nx=n, ny=max(16, n + rng.randint(-9, 9)), nz=1, call="step",
                    nsteps=rng.randint(1, 5), precision="mixed" if "mixed" in flow else "fp64")
    if flow == "layer":
        return dict(flow="layer", nx=size(100, 600), ny=size(64, 300), nz=1, call="step",
                    nsteps=rng.randint(1, 5), precision="fp64")
    if flow == "box":
        return dict(flow="box", nx=size(16, 160), ny=size(16, 160), nz=size(16, 160),
                    call=rng.choice(["rhs", "step"]), nsteps=1, precision="fp64")
    if flow == "tgv":
        n = size(24, 144)
        return dict(flow="tgv", nx=n, ny=n, nz=n, call=rng.choice(["step", "rhs", "step"]), nsteps=1,
                    precision="fp64")
    if flow == "tgv mixed":
        n = size(24, 240)
        return dict(flow="tgv", nx=n, ny=n, nz=n, call="step", nsteps=rng.randint(1, 3) if n < 128 else 1,
                    precision="mixed")
    if flow == "channel":
        return dict(flow="channel", nx=size(48, 160), ny=size(32, 128), nz=size(32, 128), call="step",
                    nsteps=1, precision="fp64")
    if flow == "porous":
        return dict(flow="porous", nx=size(96, 700), ny=size(48, 256), nz=1, call="adjoint", nsteps=1,
                    precision="fp64")
    return dict(flow="sweep", nx=size(64, 256), ny=size(64, 256), nz=size(24, 48), call="serve",
                nsteps=rng.randint(3, 10), precision=rng.choice(["fp64", "mixed"]))


def _config(case):
    """The solver's configuration of a case."""
    flow, nx, ny, nz = case["flow"], case["nx"], case["ny"], case["nz"]
    if flow == "sod":
        return wl.sod_case(nx)
    if flow in ("vortex", "riemann"):
        c = wl.vortex_case(nx) if flow == "vortex" else wl.riemann2d_case(nx)
        return dict(c, n=(nx, ny, 1))
    if flow == "layer":
        return wl.e2_case(nx, ny)
    if flow == "box":
        P = ("periodic", "periodic")
        return wl.random_box(3, (nx, ny, nz), bc=(P, ("wall", "wall"), P), visc="constant", weno="js",
                             stretch=("uniform", "tanh2", "uniform"), t_wall=((1, 1), (2.5, 2.2), (1, 1)))
    if flow == "tgv":
        return wl.tgv_case(nx)
    if flow == "channel":
        return dict(wl.channel_case(nx, ny, nz), weno="teno6a", visc_order=6)
    if flow == "porous":
        # a stable frozen step: free stream along x, sound (T up to 5) and diffusion across the wall
        c = wl.porous_bl_case(nx, ny)
        dy = float(_axes(c)[1]["dx"].min())
        return dict(c, dt_fixed=0.5 / (nx / 0.5 + 2.3 / wl.BL_MA / dy + 0.006 / (dy * dy)))
    raise ValueError(flow)


def _requests(case):
    """The solves of a serve case, as cases of their own: uneven sizes around the named ones."""
    out = []
    for k in range(8):
        f = 0.5 + 0.07 * k                                 # 0.5 .. 0.99 of the largest size
        if k % 4 == 3:
            n = max(16, int(case["nz"] * f))
            out.append(dict(flow="tgv", nx=n, ny=n, nz=n))
        else:
            out.append(dict(flow="riemann" if k % 2 else "vortex", nx=max(16, int(case["nx"] * f)),
                            ny=max(16, int(case["ny"] * f)), nz=1))
    return out


# ------------------------------------------------------------------------------------------------
# grids and initial states
# ------------------------------------------------------------------------------------------------
def _map(stretch, beta, lo, hi, eta):
    """Face coordinate x(eta) and dx/deta."""
    L = hi - lo
    if stretch == "uniform":
        return lo + L * eta, np.full_like(eta, L)
    tb = math.tanh(beta)
    t = np.tanh(beta * (2.0 * eta - 1.0)) if stretch == "tanh2" else np.tanh(beta * (1.0 - eta))
    x = lo + 0.5 * L * (1.0 + t / tb) if stretch == "tanh2" else lo + L * (1.0 - t / tb)
    return x, L * beta * (1.0 - t * t) / tb


def _axes(c):
    """Per axis over the padded range: cell centres, widths, d(index)/dx at centres and faces."""
    out = []
    for a in range(3):
        n, h = c["n"][a], H if a < c["ndim"] else 0
        i = np.arange(-h, n + h, dtype=np.float64)
        at = lambda o: _map(c["stretch"][a], c["beta"][a], c["lo"][a], c["hi"][a], (i + o) / n)  # noqa: E731
        if c["stretch"][a] == "uniform":
            d = (c["hi"][a] - c["lo"][a]) / n
            out.append(dict(n=n, h=h, xc=c["lo"][a] + (i + 0.5) * d, dx=np.full_like(i, d),
                            mc=np.full_like(i, 1.0 / d), mf=np.full_like(i, 1.0 / d)))
        else:
            lo, hi = at(0.0)[0], at(1.0)[0]
            out.append(dict(n=n, h=h, xc=0.5 * (lo + hi), dx=hi - lo, mc=n / at(0.5)[1], mf=n / at(1.0)[1]))
    return out


def _random(seed, count):
    """`count` uniform numbers in [-1, 1) of a seed (a host list)."""
    return (2.0 * np.random.default_rng(seed).random(count) - 1.0).tolist()


def _primitives(case, c, seed, device):
    """Primitives (rho, u, v, w, p) over the padded grid, made from the seed."""
    ax = _axes(c)
    x, y, z = (torch.from_numpy(ax[a]["xc"]).to(device).reshape([-1 if 2 - a == k else 1 for k in range(3)])
               for a in range(3))
    r = _random(seed, 64)
    one = torch.ones_like(x * y * z)
    flow = case["flow"]

    def waves(k, wave):
        """A smooth field of order one: three random plane waves."""
        f = 0.0
        for m in range(3):
            p = r[k + 4 * m:k + 4 * m + 4]
            f = f + p[3] * torch.sin(wave[0] * (1 + m) * x + wave[1] * (2 - m) * y + wave[2] * (1 + m) * z
                                     + math.pi * p[0])
        return f * one

    if flow == "sod":
        left = (x < 0.5 + 0.02 * r[0]) & (one > 0)
        rho = torch.where(left, 1.0 + 0.1 * r[1], 0.125 + 0.01 * r[2]) * (1 + 0.01 * torch.sin(40 * x))
        p = torch.where(left, 1.0 + 0.1 * r[3], 0.1 + 0.01 * r[4]) * one
        return torch.stack([rho, 0.05 * r[5] * torch.sin(9 * x), 0 * one, 0 * one, p])
    if flow == "vortex":
        b, dx, dy = 4.0 + r[0], x - 5.0 - 0.5 * r[1], y - 5.0 - 0.5 * r[2]
        f = torch.exp(0.5 * (1.0 - dx * dx - dy * dy)) * one
        T = 1.0 - 0.4 * b * b / (11.2 * math.pi ** 2) * f * f
        rho = T ** 2.5
        return torch.stack([rho, 1.0 - b / (2 * math.pi) * f * dy, 1.0 + b / (2 * math.pi) * f * dx, 0 * one,
                            rho * T])
    if flow == "riemann":
        q = (x >= 0.5).int() + 2 * (y >= 0.5).int() + 0 * z.int()
        v = torch.tensor(r[:16], dtype=torch.float64, device=device).reshape(4, 4)
        ripple = 1.0 + 0.02 * torch.sin(23 * x + r[16]) * torch.cos(17 * y + r[17])
        return torch.stack([(1.0 + 0.5 * v[:, 0])[q] * ripple, (0.3 * v[:, 1])[q], (0.3 * v[:, 2])[q],
                            0 * one, (0.8 + 0.4 * v[:, 3])[q] * ripple])
    if flow in ("layer", "porous"):
        # a laminar profile u = erf(y / delta) with Crocco-Busemann temperature under a weak
        # disturbance that reaches the free stream
        Ma = wl.E2_MA if flow == "layer" else wl.BL_MA
        u = torch.erf(y / (0.05 + 0.005 * r[0])) * one
        Taw = 1.0 + 0.2 * Ma * Ma
        Tw = Taw if flow == "layer" else c["t_wall"][1][0]
        T = Tw + (Taw - Tw) * u - (Taw - 1.0) * u * u
        wob = 1.0 + 0.01 * torch.sin(20 * x + 11 * y + r[1])
        return torch.stack([1.0 / T * wob, u * (1.0 + 0.01 * torch.sin(15 * x - 9 * y + r[2])),
                            0.01 * torch.tanh(8 * y) * torch.cos(12 * x + 13 * y + r[3]), 0 * one,
                            c["R"] * wob * one])
    if flow == "box":
        f = [waves(12 * k, (3.1, 2.3, 4.2)) for k in range(5)]
        return torch.stack([1.0 + 0.15 * f[0], 0.4 * f[1], 0.4 * f[2], 0.4 * f[3], 1.0 + 0.15 * f[4]])
    if flow == "tgv":
        X, Y, Z = x + r[0], y + r[1], z + r[2]
        p0 = c["T_ref"] * c["R"]
        u = torch.sin(X) * torch.cos(Y) * torch.cos(Z) + 0.05 * r[3] * torch.sin(3 * Y + 2 * Z)
        v = -torch.cos(X) * torch.sin(Y) * torch.cos(Z) + 0.05 * r[4] * torch.sin(3 * Z + 2 * X)
        w = 0.05 * r[5] * torch.sin(3 * X + 2 * Y) * one
        p = p0 + (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0) / 16.0
        return torch.stack([p / p0 * one, u, v, w, p])
    if flow == "channel":
        g = torch.Generator(device="cpu").manual_seed(seed)
        noise = 0.1 * torch.rand((3,) + tuple(one.shape), generator=g, dtype=torch.float64).to(device) - 0.05
        return torch.stack([one, 1.5 * (1.0 - y * y) * one + noise[0], noise[1], noise[2], c["R"] * one])
    raise ValueError(flow)


def _conserved(W, gamma):
    rho, u, v, w, p = W
    return torch.stack([rho, rho * u, rho * v, rho * w, p / (gamma - 1.0) + 0.5 * rho * (u * u + v * v + w * w)])


def _inputs(case, seed, device):
    """(configuration, padded state, wall parameters or None, inflow profile or None)."""
    c = _config(case)
    W = _primitives(case, c, seed, device)
    phi = inflow = None
    if case["flow"] in ("layer", "porous"):
        inflow = W[:, :, :, 0].contiguous()
    if case["flow"] == "porous":
        pz = c["porous"]
        phi = pz["phi0"] * (1.0 + 0.1 * torch.tensor(_random(seed + 1, pz["count"]), dtype=torch.float64, device=device))
    return c, _conserved(W, c["gamma"]).contiguous(), phi, inflow


def _cotangent(c, shape, seed, device):
    """A seeded cotangent of the state, zero on the halo."""
    g = torch.Generator(device="cpu").manual_seed(seed + 2)
    lam = torch.zeros(shape, dtype=torch.float64, device=device)
    i = _inner(c)
    lam[i] = (torch.rand(tuple(lam[i].shape), generator=g, dtype=torch.float64) - 0.5).to(device)
    return lam


# ------------------------------------------------------------------------------------------------
# prepare and run
# ------------------------------------------------------------------------------------------------
def prepare(case, seed):
    if case["call"] == "serve":
        from paper_2406_19494_gb300.serve import Server
        srv = Server(budget_bytes=8e9, max_active=16, chunk_steps=5)
        jobs = []
        for k, r in enumerate(_requests(case)):
            c, U, _, _ = _inputs(r, seed + 17 * k, "cpu")
            jobs.append((c, U.numpy()))
        return dict(case=case, server=srv, jobs=jobs)
    from paper_2406_19494_gb300.solver import Solver
    c, U, phi, inflow = _inputs(case, seed, "cuda")
    s = Solver(c, precision=case["precision"], adjoint=case["call"] == "adjoint")
    if phi is not None:
        s.set_wall_params(phi)
    if inflow is not None:
        s.set_inflow(0, 0, inflow)
    st = dict(case=case, solver=s, U0=U, U=U.clone())
    if case["call"] == "rhs":
        st["R"] = torch.zeros_like(U)
    if case["call"] == "adjoint":
        st["U1"], st["U2"] = torch.zeros_like(U), torch.zeros_like(U)
        end = U.clone()
        s.step_stages(end, st["U1"], st["U2"])
        st["lam0"] = _cotangent(c, U.shape, seed, "cuda")
        st["lam"] = st["lam0"].clone()
        st["gphi"] = torch.zeros_like(phi)
    return st


def run(state):
    case = state["case"]
    if case["call"] == "serve":
        srv = state["server"]
        tickets = [srv.submit(c, U, case["nsteps"], precision=case["precision"]) for c, U in state["jobs"]]
        return [srv.poll(t, timeout_ms=60000)[1] for t in tickets]
    s = state["solver"]
    if case["call"] == "rhs":
        return s.rhs(state["U0"], state["R"])
    if case["call"] == "step":
        # a new solve from its initial state
        state["U"].copy_(state["U0"])
        return s.step(state["U"], case["nsteps"])
    state["lam"].copy_(state["lam0"])
    state["gphi"].zero_()
    s.adjoint_step(state["U0"], state["lam"], gphi=state["gphi"], U1=state["U1"], U2=state["U2"])
    return {"lam": state["lam"], "gphi": state["gphi"]}


def _work_one(case, nsteps, call):
    c = _config(case)
    cells = c["n"][0] * c["n"][1] * c["n"][2]
    face = {"js": 805, "z": 845, "teno6a": 1561}[c["weno"]] + (105 if c["visc"] != "none" else 0)
    rhs = cells * c["ndim"] * face
    if call == "rhs":
        return {"bytes": 2 * 40.0 * cells, "flops": rhs}
    if call == "adjoint":
        # the three stage states and the cotangent are read, the cotangent is written; the reverse
        # of a right-hand side takes at least twice its operations
        return {"bytes": 5 * 40.0 * cells, "flops": 6 * rhs}
    # a step reads and writes its state once
    return {"bytes": nsteps * 2 * 40.0 * cells, "flops": nsteps * 3 * rhs}


def work(case):
    if case["call"] != "serve":
        return _work_one(case, case["nsteps"], case["call"])
    parts = [_work_one(r, case["nsteps"], "step") for r in _requests(case)]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


# ------------------------------------------------------------------------------------------------
# the same arithmetic in plain 64-bit torch
# ------------------------------------------------------------------------------------------------
def _inner(c):
    return (slice(None),) + tuple(slice(H if a < c["ndim"] else 0, (H if a < c["ndim"] else 0) + c["n"][a])
                                  for a in (2, 1, 0))


def _cut(f, a, lo, hi):
    return f.narrow(f.dim() - 1 - a, lo, hi - lo)


def _prims(U, c):
    rho = U[0]
    u, v, w = U[1] / rho, U[2] / rho, U[3] / rho
    p = (c["gamma"] - 1.0) * (U[4] - 0.5 * rho * (u * u + v * v + w * w))
    return torch.stack([rho, u, v, w, p, p / (rho * c["R"])])


def _with_halos(W, c, ax, phi, inflow):
    """Primitives with the halo cells of every axis in turn set by the boundary conditions; W
    covers the interior."""
    for a in range(c["ndim"]):
        n, dim, parts = c["n"][a], W.dim() - 1 - a, []
        for side in (0, 1):
            kind = c["bc"][a][side]
            if kind == "periodic":
                g = _cut(W, a, n - H, n) if side == 0 else _cut(W, a, 0, H)
            elif kind == "zero_gradient":
                e = _cut(W, a, 0, 1) if side == 0 else _cut(W, a, n - 1, n)
                g = torch.cat([e] * H, dim)
            elif kind == "inflow":
                # only the west face of the 2-D layers: the profile of the interior rows
                prof = inflow[:, :, H:H + c["n"][1]]
                prof = torch.cat([prof, (prof[4] / (prof[0] * c["R"]))[None]])
                g = torch.stack([prof] * H, -1)
            else:
                m = (_cut(W, a, 0, H) if side == 0 else _cut(W, a, n - H, n)).flip(dim)
                v = [-m[1], -m[2], -m[3]]
                if kind == "adiabatic":
                    g = torch.stack([m[0], v[0], v[1], v[2], m[4], m[5]])
                else:
                    T = 2.0 * c["t_wall"][a][side] - m[5]
                    if kind == "porous":
                        pz, x = c["porous"], ax[0]["xc"]
                        b = pz["begin"]
                        xs = torch.from_numpy(x[H + b:H + b + pz["count"]]).to(W.device)
                        vw = (pz["A"] / pz["phi0"]) * phi * torch.sin(2.0 * math.pi * pz["kappa"] * xs)
                        vw = torch.nn.functional.pad(vw, (H + b, x.size - H - b - pz["count"]))
                        v[a] = v[a] + 2.0 * vw
                    g = torch.stack([m[4] / (c["R"] * T), v[0], v[1], v[2], m[4], T])
            parts.append(g)
        W = torch.cat([parts[0], W, parts[1]], dim)
    return W


def _weno(q, kind):
    """WENO5 value at the right face of the third of five cells."""
    a, b, m, d, e = q
    p = ((2 * a - 7 * b + 11 * m) / 6, (-b + 5 * m + 2 * d) / 6, (2 * m + 5 * d - e) / 6)
    s = [13.0 / 12.0 * (x - 2 * y + z) ** 2 for x, y, z in ((a, b, m), (b, m, d), (m, d, e))]
    s[0], s[1], s[2] = (s[0] + 0.25 * (a - 4 * b + 3 * m) ** 2, s[1] + 0.25 * (b - d) ** 2,
                        s[2] + 0.25 * (3 * m - 4 * d + e) ** 2)
    if kind == "js":
        al = [w / (1e-6 + x) ** 2 for w, x in zip((0.1, 0.6, 0.3), s)]
    else:
        tau = (s[0] - s[2]).abs()
        al = [w * (1.0 + (tau / (x + 1e-40)) ** 2) for w, x in zip((0.1, 0.6, 0.3), s)]
    return (al[0] * p[0] + al[1] * p[1] + al[2] * p[2]) / (al[0] + al[1] + al[2])


def _polynomial(offsets):
    """Coefficients [m][j] of the polynomial with unit-cell averages q_j on the offsets."""
    n, half = len(offsets), Fraction(1, 2)
    M = [[((o + half) ** (m + 1) - (o - half) ** (m + 1)) / (m + 1) for m in range(n)]
         + [Fraction(int(i == j)) for j in range(n)] for i, o in enumerate(offsets)]
    for k in range(n):
        i = next(r for r in range(k, n) if M[r][k] != 0)
        M[k], M[i] = M[i], M[k]
        M[k] = [v / M[k][k] for v in M[k]]
        for r in range(n):
            if r != k:
                M[r] = [v - M[r][k] * w for v, w in zip(M[r], M[k])]
    return [row[n:] for row in M]


def _face_and_smoothness(offsets):
    """The value at x = 1/2 and the Jiang-Shu quadratic form of the offsets' polynomial."""
    n, half, C = len(offsets), Fraction(1, 2), _polynomial(offsets)
    face = [float(sum(C[m][j] * half ** m for m in range(n))) for j in range(n)]
    S = [[Fraction(0)] * n for _ in range(n)]
    for order in range(1, n):
        D = [(m - order, [math.factorial(m) // math.factorial(m - order) * v for v in C[m]]) for m in range(order, n)]
        for pa, va in D:
            for pb, vb in D:
                e = pa + pb + 1
                w = (half ** e - (-half) ** e) / e
                S = [[S[i][j] + w * va[i] * vb[j] for j in range(n)] for i in range(n)]
    return face, [[float(v) for v in row] for row in S]


_TENO = [(o, *_face_and_smoothness(o)) for o in ((-1, 0, 1), (0, 1, 2), (-2, -1, 0), (0, 1, 2, 3))]
_TENO6 = _face_and_smoothness((-2, -1, 0, 1, 2, 3))[1]


def _form(S, q):
    d = [v - q[0] for v in q]
    return sum(S[i][j] * d[i] * d[j] for i in range(len(q)) for j in range(len(q)) if S[i][j])


def _teno(q):
    """TENO6-A value at the right face of the third of six cells."""
    p = [sum(f * q[o + 2] for f, o in zip(face, off)) for off, face, _ in _TENO]
    b = [_form(S, [q[o + 2] for o in off]) for off, _, S in _TENO]
    tau = (_form(_TENO6, q) - (b[1] + b[2] + 4.0 * b[0]) / 6.0).abs()
    g = [(1.0 + tau / (x + 1e-40)) ** 6 for x in b]
    e = 0.9 * 0.25 * 1e-6 / 0.75
    D = [q[j + 1] - q[j] for j in range(5)]
    eta = None
    for j in range(4):
        s = (2.0 * (D[j + 1] * D[j]).abs() + e) / (D[j + 1] ** 2 + D[j] ** 2 + e)
        eta = s if eta is None else torch.minimum(eta, s)
    m = 1.0 - (eta / 0.25).clamp(max=1.0)
    ct = 10.0 ** -torch.floor(10.5 - 3.5 * (1.0 - (1.0 - m) ** 4 * (1.0 + 4.0 * m)))
    tot = g[0] + g[1] + g[2] + g[3]
    w = [d * (~(x / tot < ct)).double() for d, x in zip((0.45, 0.3, 0.05, 0.2), g)]
    return sum(x * y for x, y in zip(w, p)) / (w[0] + w[1] + w[2] + w[3])


def _hllc(L, R, d, gamma):
    def side(W):
        q2 = W[1] ** 2 + W[2] ** 2 + W[3] ** 2
        E = W[4] / (gamma - 1.0) + 0.5 * W[0] * q2
        U = [W[0], W[0] * W[1], W[0] * W[2], W[0] * W[3], E]
        F = [W[1 + d] * x for x in U]
        F[1 + d] = F[1 + d] + W[4]
        F[4] = F[4] + W[1 + d] * W[4]
        return U, F, torch.sqrt(gamma * W[4] / W[0]), (E + W[4]) / W[0], torch.sqrt(W[0])

    UL, FL, cL, HL, sL = side(L)
    UR, FR, cR, HR, sR = side(R)
    v = [(sL * L[1 + k] + sR * R[1 + k]) / (sL + sR) for k in range(3)]
    Ht = (sL * HL + sR * HR) / (sL + sR)
    ct = torch.sqrt((gamma - 1.0) * (Ht - 0.5 * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2)))
    SL = torch.minimum(L[1 + d] - cL, v[d] - ct)
    SR = torch.maximum(R[1 + d] + cR, v[d] + ct)
    mL, mR = L[0] * (SL - L[1 + d]), R[0] * (SR - R[1 + d])
    S = (R[4] - L[4] + L[1 + d] * mL - R[1 + d] * mR) / (mL - mR)

    def star(W, U, F, SK, m):
        fac = m / (SK - S)
        X = [fac, fac * W[1], fac * W[2], fac * W[3],
             fac * (U[4] / W[0] + (S - W[1 + d]) * (S + W[4] / m))]
        X[1 + d] = fac * S
        return [f + SK * (x - u) for f, x, u in zip(F, X, U)]

    ls, rs = star(L, UL, FL, SL, mL), star(R, UR, FR, SR, mR)
    return [torch.where(SL >= 0, FL[k], torch.where(S >= 0, ls[k], torch.where(SR > 0, rs[k], FR[k])))
            for k in range(5)]


def _mu(T, c):
    r = T / c["T_ref"]
    if c["visc"] == "constant":
        return c["mu_ref"] * torch.ones_like(T)
    if c["visc"] == "power":
        return c["mu_ref"] * r ** c["visc_exp"]
    return c["mu_ref"] * r ** 1.5 * (c["T_ref"] + c["suth_S"]) / (T + c["suth_S"])


def _along(v, a, device):
    return torch.from_numpy(v).to(device).reshape([-1 if 2 - a == k else 1 for k in range(3)])


def _dissipative(W, c, ax, d):
    six = c.get("visc_order", 4) == 6
    n, dev = c["n"][d], W.device
    at = lambda f, o: _cut(f, d, H - 1 + o, H + n + o)  # noqa: E731
    if six:
        ip = lambda f: (150.0 * (at(f, 0) + at(f, 1)) - 25.0 * (at(f, -1) + at(f, 2)) + 3.0 * (at(f, -2) + at(f, 3))) / 256.0  # noqa: E731,E501
        dn = lambda f: (2250.0 * (at(f, 1) - at(f, 0)) - 125.0 * (at(f, 2) - at(f, -1)) + 9.0 * (at(f, 3) - at(f, -2))) / 1920.0  # noqa: E731,E501
    else:
        ip = lambda f: (9.0 * (at(f, 0) + at(f, 1)) - (at(f, -1) + at(f, 2))) / 16.0  # noqa: E731
        dn = lambda f: ((at(f, -1) - at(f, 2)) + 27.0 * (at(f, 1) - at(f, 0))) / 24.0  # noqa: E731
    mf = _along(ax[d]["mf"][H - 1:H + n], d, dev)

    def centre(f, b):
        nb = f.shape[2 - b]
        s = lambda o: _cut(f, b, 3 + o, nb - 3 + o)  # noqa: E731
        if six:
            g = (45.0 * (s(1) - s(-1)) - 9.0 * (s(2) - s(-2)) + (s(3) - s(-3))) / 60.0
        else:
            g = ((s(-2) - s(2)) + 8.0 * (s(1) - s(-1))) / 12.0
        return g * _along(ax[b]["mc"][3:nb - 3], b, dev)

    def tang(f, skip=None):
        for b in range(c["ndim"]):
            if b not in (d, skip):
                f = _cut(f, b, H, H + c["n"][b])
        return f

    v = [tang(ip(W[1 + k])) for k in range(3)]
    G = [[torch.zeros_like(v[0]) for _ in range(3)] for _ in range(3)]
    for k in range(3):
        G[k][d] = tang(dn(W[1 + k])) * mf
    for b in range(c["ndim"]):
        if b != d:
            G[d][b] = ip(centre(tang(W[1 + d], b), b))
            G[b][b] = ip(centre(tang(W[1 + b], b), b))
    div = G[0][0] + G[1][1] + G[2][2]
    mu = _mu(tang(ip(W[5])), c)
    tau = [mu * (G[k][d] + G[d][k]) - ((2.0 / 3.0) * mu * div if k == d else 0.0) for k in range(3)]
    cp = c["gamma"] * c["R"] / (c["gamma"] - 1.0)
    return tau + [v[0] * tau[0] + v[1] * tau[1] + v[2] * tau[2] + mu * (cp / c["Pr"]) * tang(dn(W[5])) * mf]


def _rhs(U, c, ax, phi, inflow):
    """dU/dt of the interior from the interior state."""
    W = _with_halos(_prims(U, c), c, ax, phi, inflow)
    R = torch.zeros_like(U)
    for d in range(c["ndim"]):
        n, V = c["n"][d], W
        for b in range(c["ndim"]):
            if b != d:
                V = _cut(V, b, H, H + c["n"][b])
        at = lambda k, o: _cut(V[k], d, H - 1 + o, H + n + o)  # noqa: E731
        if c["weno"] == "teno6a":
            L = [_teno([at(k, o) for o in range(-2, 4)]) for k in range(5)]
            Q = [_teno([at(k, o) for o in range(3, -3, -1)]) for k in range(5)]
            for S, o in ((L, 0), (Q, 1)):
                bad = (S[0] <= 0) | (S[4] <= 0)
                S[:] = [torch.where(bad, at(k, o), S[k]) for k in range(5)]
        else:
            L = [_weno([at(k, o) for o in range(-2, 3)], c["weno"]) for k in range(5)]
            Q = [_weno([at(k, o) for o in range(3, -2, -1)], c["weno"]) for k in range(5)]
        F = _hllc(L, Q, d, c["gamma"])
        if c["visc"] != "none":
            Fd = _dissipative(W, c, ax, d)
            F = [F[0]] + [f - g for f, g in zip(F[1:], Fd)]
        F = torch.stack(F)
        R = R - (_cut(F, d, 1, n + 1) - _cut(F, d, 0, n)) / _along(ax[d]["dx"][H if n > 1 else 0:][:n], d, U.device)
    f = c["body_force"]
    if any(f):
        u = [U[1 + k] / U[0] for k in range(3)]
        zero = torch.zeros_like(u[0])
        R = R + torch.stack([zero] + [zero + f[k] for k in range(3)] + [f[0] * u[0] + f[1] * u[1] + f[2] * u[2]])
    return R


def _dt(U, c, ax):
    if c["dt_fixed"] > 0:
        return c["dt_fixed"]
    W, best = _prims(U, c), math.inf
    a = torch.sqrt(c["gamma"] * W[4] / W[0])
    for d in range(c["ndim"]):
        dx = _along(ax[d]["dx"][H:H + c["n"][d]], d, U.device)
        best = min(best, float((dx / (W[1 + d].abs() + a)).min()))
        if c["visc"] != "none":
            k = 2.0 * max(4.0 / 3.0, c["gamma"] / c["Pr"])
            best = min(best, float((dx * dx / (k * _mu(W[5], c) / W[0])).min()))
    return c["cfl"] * best


def _exact_step(U, c, ax, phi, inflow, nsteps):
    for _ in range(nsteps):
        dt = _dt(U, c, ax)
        U1 = U + dt * _rhs(U, c, ax, phi, inflow)
        U2 = 0.75 * U + 0.25 * (U1 + dt * _rhs(U1, c, ax, phi, inflow))
        U = U / 3.0 + (2.0 / 3.0) * (U2 + dt * _rhs(U2, c, ax, phi, inflow))
    return U


def _exact_adjoint(U0, c, ax, phi, inflow, lam):
    """The transposed step, stage by stage, with the stage states formed in 64 bits."""
    dt, gphi = c["dt_fixed"], torch.zeros_like(phi)
    with torch.no_grad():
        U1 = U0 + dt * _rhs(U0, c, ax, phi, inflow)
        U2 = 0.75 * U0 + 0.25 * (U1 + dt * _rhs(U1, c, ax, phi, inflow))

    def back(X, mu):
        X, p = X.detach().requires_grad_(True), phi.detach().requires_grad_(True)
        gX, gp = torch.autograd.grad(_rhs(X, c, ax, p, inflow), (X, p), mu)
        gphi.add_(gp)
        return gX

    l2 = (2.0 / 3.0) * lam + back(U2, (2.0 / 3.0) * dt * lam)
    l1 = 0.25 * l2 + back(U1, 0.25 * dt * l2)
    return lam / 3.0 + 0.75 * l2 + l1 + back(U0, dt * l1), gphi


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["call"] == "serve":
        out = []
        for k, r in enumerate(_requests(case)):
            c, U, _, _ = _inputs(r, seed + 17 * k, dev)
            i = _inner(c)
            U[i] = _exact_step(U[i], c, _axes(c), None, None, case["nsteps"])
            out.append(U.cpu().numpy())
        return out
    c, U, phi, inflow = _inputs(case, seed, dev)
    ax, i = _axes(c), _inner(c)
    if case["call"] == "adjoint":
        lam = _cotangent(c, U.shape, seed, dev)
        lam[i], gphi = _exact_adjoint(U[i], c, ax, phi, inflow, lam[i])
        return {"lam": lam, "gphi": gphi}
    if case["call"] == "rhs":
        R = torch.zeros_like(U)
        R[i] = _rhs(U[i], c, ax, phi, inflow)
        return R
    U[i] = _exact_step(U[i], c, ax, phi, inflow, case["nsteps"])
    return U

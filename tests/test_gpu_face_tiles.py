"""The FP64 face kernels' tiles against the oracle at the sizes where they can go wrong: lines one cell
shorter, equal to and longer than a tile's cells (27 along y and z, 123 along x), the shortest lines, ragged
columns, and states on both sides of the two-float path's limits (smooth waves and grid-scale noise of
growing size, strong and weak dissipation).

Tolerance: a face flux is formed with at most 32 roundings of its own size, the primitives with 8, and R
is a difference of two of them over dx on each axis, so |R - R_oracle| <= 2 ndim 80 2^-53 S / dx, S the
largest of rho (|u| + c), rho (|u| + c)^2 and rho (|u| + c)^3 (with the dissipative fluxes added to it)."""
import numpy as np
import pytest

from oracle import ns_fv as nf
from paper_2406_19494_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
P = ("periodic", "periodic")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_19494_gb300 import build
    build.build()


def check(n, amp, kind, **kw):
    from paper_2406_19494_gb300.solver import Solver
    ndim = 1 + (n[1] > 1) + (n[2] > 1)
    kw.setdefault("visc", "power")
    c = wl.random_box(ndim, n, bc=(P, P, P), hi=tuple(lo + 0.1 * k for lo, k in zip((0.0, -1.0, 0.0), n)), **kw)
    case = nf.Case(c)
    grid = nf.Grid(case)
    rng = np.random.default_rng(7 * n[0] + n[1] + int(1e6 * amp) % 997)
    W = np.empty(case.shape)
    base = (1.0, 0.2, -0.1, 0.3, 0.9)
    i = [np.arange(case.p[a]) - case.h[a] for a in (2, 1, 0)]
    z, y, x = np.meshgrid(*i, indexing="ij")
    for v in range(5):
        if kind == "noise":
            f = rng.uniform(-1, 1, case.shape[1:])
        else:
            ph = rng.uniform(0, 6.28, 4)
            f = np.sin(0.4 * x + ph[0]) * np.cos(0.3 * y + ph[1]) * np.cos(0.5 * z + ph[2])
        W[v] = base[v] + amp * f
    U = nf.prim_to_cons(W, case)
    R_ref = nf.rhs(U.copy(), case, grid)
    s = Solver(c)
    R = s.rhs(torch.from_numpy(U).cuda())
    s.check()
    inner = (slice(None),) + case.interior()
    err = np.abs(R.cpu().numpy()[inner] - R_ref[inner])
    cs = np.sqrt(1.4 * (W[4] / W[0]).max())
    sp = np.abs(W[1:4]).max() + cs
    visc = 0.0 if c["visc"] == "none" else 4.0 * c["mu_ref"] * amp / 0.1 * (3.5 / 0.72 + sp)
    S = W[0].max() * max(sp, sp ** 2, sp ** 3) + visc
    assert err.max() <= 2 * ndim * 80 * 2.0 ** -53 * S / 0.1, (err.max(), S)


@pytest.mark.parametrize("n", [(3, 3, 3), (117, 3, 1), (123, 4, 1), (124, 5, 1), (9, 21, 3), (8, 27, 5),
                               (7, 28, 3), (17, 3, 27), (15, 4, 55), (250, 1, 1)])
def test_tile_edges(n):
    check(n, 0.02, "wave")
    check(n, 0.2, "noise", weno="js", visc="none")
    check(n, 0.1, "noise", weno="teno6a", visc_order=6)


@pytest.mark.parametrize("kind", ["wave", "noise"])
@pytest.mark.parametrize("amp", [1e-7, 1e-4, 1e-3, 3e-3, 1e-2, 0.1, 0.4])
def test_limits_of_the_two_float_path(amp, kind):
    check((33, 30, 4), amp, kind)
    check((33, 30, 4), amp, kind, weno="js", visc="sutherland", mu_ref=1e-4)
    check((33, 30, 4), amp, kind, weno="teno6a", visc_order=6, mu_ref=1e-3)

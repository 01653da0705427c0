"""The adjoint of a right-hand side where its cotangent is zero, or too small for the two-float forms'
scaling.  R at a cell depends on the cells within three along each axis and, through the tangential
gradients, on those within three along one axis and two along another, so the gradient is exactly zero
outside that box; it is linear in the cotangent, and the two-float and FP64 forms of its faces differ by
less than 1e-10 of the largest entry (the adjoint tests' bound)."""
import numpy as np
import pytest

from helpers import padded_state
from paper_2406_19494_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P = ("periodic", "periodic")
WALL = dict(bc=(P, ("wall", "wall"), P), t_wall=((1, 1), (2.5, 2.2), (1, 1)))


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_19494_gb300 import build
    build.build()


def _adjoint(c, U, mu):
    from paper_2406_19494_gb300.solver import Solver
    return Solver(c, adjoint=True).adjoint_rhs(torch.from_numpy(U).cuda(), torch.from_numpy(mu).cuda()).cpu().numpy()


@pytest.mark.parametrize("kw", [WALL, dict(weno="js", visc="none"), dict(bc=(P, P, P), visc="constant")])
def test_a_zero_cotangent_gives_a_zero_gradient(kw):
    c = wl.random_box(2, (45, 19, 1), **kw)
    _, _, U = padded_state(c, seed=3)
    assert np.array_equal(_adjoint(c, U, np.zeros_like(U)), np.zeros_like(U))


@pytest.mark.parametrize("n,at", [((45, 37, 1), (20, 18, 0)), ((21, 20, 19), (10, 9, 9))])
@pytest.mark.parametrize("v", [0, 2, 4])
def test_a_local_cotangent_reaches_its_stencil_only(n, at, v):
    ndim = 3 if n[2] > 1 else 2
    c = wl.random_box(ndim, n, **WALL)
    case, _, U = padded_state(c, seed=3)
    h = case.h
    mu = np.zeros_like(U)
    mu[v, h[2] + at[2], h[1] + at[1], h[0] + at[0]] = 0.7
    g = _adjoint(c, U, mu)
    box = tuple(slice(h[a] + at[a] - 3, h[a] + at[a] + 4) if n[a] > 1 else slice(None) for a in (2, 1, 0))
    assert np.abs(g[(slice(None),) + box]).max() > 0
    g[(slice(None),) + box] = 0.0
    assert np.array_equal(g, np.zeros_like(g))


@pytest.mark.parametrize("k", [-1000, -960, 890, 950])
def test_cotangents_beyond_the_scaling_take_fp64(k):
    c = wl.random_box(2, (40, 15, 1), **WALL)
    case, _, U = padded_state(c, seed=4)
    inner = (slice(None),) + case.interior()
    mu = np.zeros_like(U)
    mu[inner] = np.random.default_rng(6).uniform(-1, 1, mu[inner].shape)
    mu[2] = 0.0
    a, b = _adjoint(c, U, mu)[inner], _adjoint(c, U, np.ldexp(mu, k))[inner]
    for i in range(5):
        # below 2^-1022 the result is a subnormal number
        assert np.abs(np.ldexp(b[i], -k) - a[i]).max() <= 1e-10 * np.abs(a[i]).max() + np.ldexp(1.0, max(-1074 - k, -1074) + 20) * (k < -950)

"""Two-float adjoint faces: the edges of their tiles and their way back to FP64.

The adjoint of one right-hand side against complex-step derivatives of the CPU oracle, which are exact
to rounding, at sizes around the tiles (31 faces along x, 7 along y and z, 8 or 32 lines across); the
bound is the adjoint tests' 1e-10 of the summed terms.  A state times 2^60 (with the viscosity) has the
same Jacobian, but leaves the range of the two floats, so every face takes FP64: against the unscaled
state each entry may differ by the two sides' errors, below 1e-10 of the largest.  A cotangent times a
power of two gives the same bits times that power.
"""
import numpy as np
import pytest

from helpers import padded_state
from oracle import ns_fv as nf
from paper_2406_19494_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H = 1e-30
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


def _cotangent(case, rng, shape):
    X = np.zeros(shape)
    inner = (slice(None),) + case.interior()
    X[inner] = rng.uniform(-1, 1, X[inner].shape)
    return X


@pytest.mark.parametrize("n,kw", [
    ((29, 6, 1), dict(visc="sutherland")), ((30, 7, 1), dict(weno="js")), ((31, 8, 1), dict(visc="constant")),
    ((33, 13, 1), WALL), ((62, 14, 1), dict(WALL, weno="js")), ((63, 5, 1), dict(visc="none")),
    ((32, 9, 6), dict(visc="sutherland")), ((5, 7, 7), WALL), ((33, 6, 15), dict(weno="js")),
])
def test_tile_edges_match_complex_step(n, kw):
    c = wl.random_box(3 if n[2] > 1 else 2, n, **kw)
    case, grid, U = padded_state(c, seed=n[0])
    rng = np.random.default_rng(n[1])
    mu = _cotangent(case, rng, U.shape)
    dU = _cotangent(case, rng, U.shape) * np.abs(U).max(axis=(1, 2, 3))[:, None, None, None] * 0.1
    d = nf.rhs((U + 1j * H * dU).copy(), case, grid, None, {}).imag / H
    inner = (slice(None),) + case.interior()
    gU = _adjoint(c, U, mu)
    assert abs(np.sum(mu * d) - np.sum(gU[inner] * dU[inner])) <= 1e-10 * np.sum(np.abs(mu * d))


@pytest.mark.parametrize("weno", ["z", "js"])
@pytest.mark.parametrize("visc", ["none", "constant"])
def test_states_beyond_the_two_floats_take_fp64(weno, visc):
    f = 2.0 ** 60
    c = wl.random_box(2, (45, 17, 1), weno=weno, visc=visc, weno_eps=1e-40)
    big = dict(c, mu_ref=c["mu_ref"] * f)
    case, _, U = padded_state(c, seed=2)
    mu = _cotangent(case, np.random.default_rng(5), U.shape)
    a, b = _adjoint(c, U, mu), _adjoint(big, U * f, mu)
    inner = (slice(None),) + case.interior()
    for v in range(5):
        assert np.abs(a[v][inner[1:]] - b[v][inner[1:]]).max() <= 1e-10 * np.abs(b[v][inner[1:]]).max()


@pytest.mark.parametrize("k", [-900, -200, -40, 60, 300, 800])
def test_cotangents_of_any_size(k):
    c = wl.random_box(2, (40, 15, 1), **WALL)
    case, _, U = padded_state(c, seed=4)
    mu = _cotangent(case, np.random.default_rng(6), U.shape)
    inner = (slice(None),) + case.interior()
    a, b = _adjoint(c, U, mu)[inner], _adjoint(c, U, np.ldexp(mu, k))[inner]
    assert np.array_equal(np.ldexp(a, k), b)

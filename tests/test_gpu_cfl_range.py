"""The CFL time step where a cell's p / rho leaves the FP32 range, so that its FP32 rate says nothing: the
cell must still count.  The step is cfl over the largest (|u| + c) / dx: ten FP64 roundings, and at the
fast cell those of its pressure, 2^-53 E / p = 2e-7 of a sound speed 1e-5 of u, hence 1e-11."""
import numpy as np
import pytest

from oracle import ns_fv as nf
from paper_2406_19494_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_19494_gb300 import build
    build.build()


# (rho, u, p) of most cells and of one cell with the largest rate: sound speed 1.2e21 among 1.2;
# speed 1e-18 with p / rho = 1e-46 among sound speeds of 3.7e-19
@pytest.mark.parametrize("base,one", [((1.0, 0.0, 1.0), (1e-25, 0.0, 1e17)), ((1e20, 0.0, 1e-17), (1e20, 1e-18, 1e-26))])
@pytest.mark.parametrize("at", [0, 255, 256, 299])
def test_a_cell_outside_the_fp32_range_counts(base, one, at):
    from paper_2406_19494_gb300.solver import Solver
    c = wl.random_box(1, (300, 1, 1), visc="none")
    case = nf.Case(c)
    W = np.zeros(case.shape)
    for v, a, b in zip((0, 1, 4), base, one):
        W[v] = a
        W[v, :, :, case.h[0] + at] = b
    U = nf.prim_to_cons(W, case)
    s = Solver(c)
    dt = s.compute_dt(torch.from_numpy(U).cuda()).item()
    s.check()
    rho, m, E = U[0, 0, 0], U[1, 0, 0], U[4, 0, 0]
    p = (case.gamma - 1.0) * (E - 0.5 * m * m / rho)
    dx = (c["hi"][0] - c["lo"][0]) / 300
    ref = c["cfl"] * dx / (np.abs(m / rho) + np.sqrt(case.gamma * p / rho)).max()
    assert abs(dt - ref) <= 1e-11 * ref

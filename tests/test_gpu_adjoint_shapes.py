"""The discrete adjoint on ragged lattices and every boundary rule, where the
reverse kernel's 60-node segments, row ends and wall rows can go wrong: the
gradient against central differences (eps = 1e-4) of the FP64 oracle, along the
marker gradient's own direction and for the inflow speed, over a window of 40
steps from the initial fields (checkpoint every 16: a ragged last segment).  Bar:
1e-3 relative, the one of the 160 x 80 comparison."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1806_09403_gb300 import _build  # noqa: E402
from paper_1806_09403_gb300 import btdf as B  # noqa: E402

STEPS, EVERY, EPS, TOL = 40, 16, 1e-4, 1e-3


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()


def case(nx, ny, bcx, bcy, delta):
    c = W.Case("adj", nx, ny, 0.6, 0.05, delta, bcx, bcy, seed=nx, D=8.0)
    # the second body's support reaches the last strip's border columns and the rows by a wall
    c.bodies.append(W.circle_markers(0.4 * nx, 0.5 * ny + 0.2, 8.0, 25))
    c.bodies.append(W.circle_markers(nx - 10.3, 8.2, 8.0, 25))
    return c


def oracle_J(c, fields, X, Y, u):
    s = O.Sim(c.nx, c.ny, c.tau, u, c.bc_x, c.bc_y, delta=c.delta)
    s.init_fields(*fields)
    n = 0
    for b in c.bodies:
        m = len(b.X)
        s.add_body(X[n:n + m], Y[n:n + m], b.ds)
        n += m
    s.step(STEPS)
    fx = sum(s.history(k, 0, STEPS)[0] for k in range(len(c.bodies)))
    return float(fx.mean() / (0.5 * u * u * c.D))


@pytest.mark.parametrize("bcx,bcy", [(W.BCX_INOUT, W.BCY_FREESLIP), (W.BCX_INOUT, W.BCY_NOSLIP),
                                     (W.BCX_INOUT, W.BCY_PERIODIC), (W.BCX_PERIODIC, W.BCY_PERIODIC),
                                     (W.BCX_PERIODIC, W.BCY_NOSLIP)])
@pytest.mark.parametrize("nx,ny,delta", [(59, 33, 4), (60, 34, 5), (61, 33, 3), (62, 37, 4), (121, 41, 4)])
def test_adjoint_against_fp64_differences(nx, ny, delta, bcx, bcy):
    c = case(nx, ny, bcx, bcy, delta)
    fields = c.initial_fields()
    lat = B.Lattice.from_case(c)
    J = lat.adjoint_forward(STEPS, EVERY, -1, c.D)
    dU, dX, dY = lat.adjoint_backward()
    X, Y = (np.concatenate([getattr(b, k) for b in c.bodies]) for k in "XY")
    assert abs(J / oracle_J(c, fields, X, Y, c.u_in) - 1) <= 1e-4
    norm = np.sqrt((dX ** 2 + dY ** 2).sum())
    vx, vy = dX / norm, dY / norm
    fd = (oracle_J(c, fields, X + EPS * vx, Y + EPS * vy, c.u_in)
          - oracle_J(c, fields, X - EPS * vx, Y - EPS * vy, c.u_in)) / (2 * EPS)
    print(f"\n{nx}x{ny} bcx {bcx} bcy {bcy}: |dJ/dX| {norm:.6e} (FD {fd:.6e}, {abs(norm / fd - 1):.1e}); "
          f"J {J:.6f}", end="")
    assert abs(norm / fd - 1) <= TOL
    fdU = (oracle_J(c, fields, X, Y, c.u_in + EPS) - oracle_J(c, fields, X, Y, c.u_in - EPS)) / (2 * EPS)
    print(f"; dJ/dU {dU:.6e} (FD {fdU:.6e}, {abs(dU / fdU - 1):.1e})", end="")
    assert abs(dU / fdU - 1) <= TOL
    lat.close()

"""Two steps per pass (the pair kernels) against single steps of variant 1: the
same arithmetic node by node, so populations, marker results and body forces are
equal bit for bit.  Sizes sit at the edges of the kernel's tiles (30 lanes of 2
or 4 nodes, 6 or 7 rows) and of the vectors; bodies reach the walls, wrap around
periodic edges and straddle tiles.  FP32 takes 2 nodes per lane below 2^22 nodes:
its 4-node form is covered where nx - 1 starts a 60-node tile."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1806_09403_gb300 import _build  # noqa: E402
from paper_1806_09403_gb300 import btdf as B  # noqa: E402

STORAGES = [B.BTDF_F32, B.BTDF_F16DEV, B.BTDF_BF16DEV]


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()


def case(nx, ny, bcx, bcy, delta=3, bodies=(), gx=0.0, tau=0.6):
    c = W.Case("pair", nx, ny, tau, 0.04, delta, bcx, bcy, seed=nx + ny, noise=1e-3, gx=gx)
    for cx, cy, d in bodies:
        b = W.circle_markers(cx, cy, d, max(6, int(np.pi * d)))
        b.Ubx[:] = 0.01
        c.bodies.append(b)
    return c


# Pairs start once enough steps of the same markers make up for their tables
# (64, or one call of as many); every run below ends with pairs in short calls.
def compare(c, storage, layout=None, steps=(1, 2, 66, 2, 5)):
    a = B.Lattice.from_case(c, storage=storage, layout=layout, history_len=16)
    b = B.Lattice.from_case(c, storage=storage, layout=layout, history_len=16)
    b.tune(1)
    for n in steps:
        a.step(n)
        b.step(n)
        assert np.array_equal(a.field(B.FIELD_POPS), b.field(B.FIELD_POPS)), (n, a.steps)
        for k in range(len(c.bodies)):
            m, r = a.markers(k), b.markers(k)
            assert all(np.array_equal(m[q], r[q]) for q in m)
            fa, fb = (x.forces(k, x.steps - min(n, 8), min(n, 8)) for x in (a, b))
            assert np.array_equal(fa[0], fb[0]) and np.array_equal(fa[1], fb[1])
    if c.bodies:   # marker velocities and the force field belong to the last step
        assert np.array_equal(a.field(B.FIELD_FX), b.field(B.FIELD_FX))
    a.close()
    b.close()


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("bcx,bcy", [(W.BCX_INOUT, W.BCY_FREESLIP), (W.BCX_PERIODIC, W.BCY_PERIODIC),
                                     (W.BCX_CONVECTIVE, W.BCY_NOSLIP), (W.BCX_PERIODIC, W.BCY_NOSLIP)])
@pytest.mark.parametrize("nx", [118, 119, 120, 121, 122, 124, 128, 129, 240, 241, 363])
def test_strip_edges(nx, bcx, bcy, storage):
    ny = 37
    bodies = [(nx - 22.3, 18.4, 9.0), (15.2, 20.1, 7.0)]
    if bcx == W.BCX_PERIODIC:
        bodies.append((0.3, 12.0, 6.0))            # wraps in x
    compare(case(nx, ny, bcx, bcy, bodies=bodies, gx=1e-6 if bcx == W.BCX_PERIODIC else 0.0), storage)


@pytest.mark.parametrize("ny", [4, 5, 7, 31, 32, 33, 64, 65, 97])
@pytest.mark.parametrize("bcy", [W.BCY_PERIODIC, W.BCY_FREESLIP, W.BCY_NOSLIP])
def test_row_edges(ny, bcy):
    for bcx, nx in ((W.BCX_INOUT, 64), (W.BCX_PERIODIC, 33), (W.BCX_PERIODIC, 4), (W.BCX_INOUT, 5)):
        compare(case(nx, ny, bcx, bcy), B.BTDF_F32)


@pytest.mark.parametrize("delta", [2, 3, 4, 5])
@pytest.mark.parametrize("layout", [B.LAYOUT_ROWS, B.LAYOUT_PLANES])
def test_deltas_walls_and_layouts(delta, layout):
    # bodies resting on the wall rows, on a strip border (x = 120) and across the periodic y edge
    r = {2: 5.0, 3: 5.5, 4: 6.0, 5: 6.0}[delta]
    ny = 70
    wall = [(60.3, r + 0.6, 10.0), (120.2, 40.0, 12.0), (200.7, ny - 1 - r, 10.0)]
    for bcy in (W.BCY_FREESLIP, W.BCY_NOSLIP):
        compare(case(250, ny, W.BCX_INOUT, bcy, delta, wall, tau=1.5), B.BTDF_F32, layout)
    wrap = [(60.3, 0.4, 10.0), (120.2, 40.0, 12.0), (249.6, 69.7, 8.0)]
    compare(case(250, 70, W.BCX_PERIODIC, W.BCY_PERIODIC, delta, wrap, tau=1.5), B.BTDF_F16DEV, layout)


def test_clipped_supports_take_single_steps():
    # a marker 0.3 above row 0: its support is cut, so the pair path must not be taken
    compare(case(96, 48, W.BCX_INOUT, W.BCY_FREESLIP, 3, [(40.0, 4.3, 8.0)], tau=1.0), B.BTDF_F32)


def test_larger_lattice_and_many_bodies():
    bodies = [(40.0 + 37.0 * i + 0.31 * j, 30.0 + 33.0 * j + 0.17 * i, 14.0) for i in range(12) for j in range(8)]
    for storage in STORAGES:
        compare(case(499, 301, W.BCX_INOUT, W.BCY_FREESLIP, 3, bodies), storage, steps=(2, 131, 4))


@pytest.mark.parametrize("storage", STORAGES)
def test_many_inlet_and_outlet_nodes(storage):
    # roundings of the row ends that differ once in thousands of nodes
    for bcx in (W.BCX_INOUT, W.BCX_CONVECTIVE):
        compare(case(90, 4001, bcx, W.BCY_FREESLIP, tau=0.53, bodies=[(45.0, 2000.0, 9.0)]), storage, steps=(1, 130))


@pytest.mark.parametrize("storage", STORAGES)
def test_batch_pairs(storage):
    """The batch's pairs (automatic shape) against launch shape 1, which steps
    singly: lattices of both strip widths' edges, every boundary kind, with and
    without bodies."""
    cases = [case(nx, ny, bcx, bcy, bodies=bodies, gx=1e-6 if bcx == W.BCX_PERIODIC else 0.0)
             for nx, ny, bcx, bcy, bodies in [
                 (121, 37, W.BCX_INOUT, W.BCY_FREESLIP, [(100.0, 18.4, 9.0), (15.2, 20.1, 7.0)]),
                 (64, 29, W.BCX_PERIODIC, W.BCY_PERIODIC, [(0.3, 12.0, 6.0)]),
                 (119, 30, W.BCX_PERIODIC, W.BCY_NOSLIP, [(40.0, 15.0, 8.0)]),
                 (48, 36, W.BCX_INOUT, W.BCY_NOSLIP, []),
                 (250, 64, W.BCX_INOUT, W.BCY_PERIODIC, [(120.3, 30.0, 12.0)])]]
    a = B.Batch.from_cases(cases, storage=storage, history_len=16)
    b = B.Batch.from_cases(cases, storage=storage, history_len=16)
    b.tune(1)
    for n in (1, 2, 5, 66):
        a.step(n)
        b.step(n)
        for i in range(len(cases)):
            assert np.array_equal(a.field(i, B.FIELD_POPS), b.field(i, B.FIELD_POPS)), (n, i)
        for k in range(len(a.bodies)):
            fa, fb = (x.forces(k, x.steps - min(n, 8), min(n, 8)) for x in (a, b))
            assert np.array_equal(fa[0], fb[0]) and np.array_equal(fa[1], fb[1]), (n, k)


def test_history_of_one_step_and_moved_markers():
    # a ring of one step keeps the last step's forces; moved markers rebuild the tables
    c = case(150, 61, W.BCX_INOUT, W.BCY_FREESLIP, bodies=[(60.3, 30.2, 9.0)])
    a = B.Lattice.from_case(c, history_len=1)
    b = B.Lattice.from_case(c, history_len=1)
    b.tune(1)
    for move, n in ((0.0, 80), (0.4, 2), (0.4, 70), (0.9, 3), (0.9, 64), (0.9, 4)):
        for x in (a, b):
            if move:
                x.move_markers(0, c.bodies[0].X + move, c.bodies[0].Y)
            x.step(n)
        fa, fb = a.forces(0, a.steps - 1, 1), b.forces(0, b.steps - 1, 1)
        assert np.array_equal(fa[0], fb[0]) and np.array_equal(fa[1], fb[1])
        assert np.array_equal(a.field(B.FIELD_POPS), b.field(B.FIELD_POPS))

"""Paired steps against single steps over everything that the rule for pairs
accepts: strip and tile widths, boundary kinds, deltas, storages, layouts, forces,
short history rings, inflow changes, checkpoints and moved markers between calls.
Both sides round alike, so populations, marker results and forces are equal bit
for bit."""
import random

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


def lattices(nx, ny, storage, bcx, bcy, bodies=(), delta=3, u=0.05, gx=0.0, gy=0.0, tau=0.6, layout=None, hist=64):
    """The same lattice twice: steps chosen by the library, and single steps."""
    rng = np.random.default_rng(nx * 1000 + ny)
    rho, ux, uy = (c + 1e-3 * rng.standard_normal((ny, nx)) for c in (1.0, u, 0.0))
    pair = []
    for _ in range(2):
        x = B.Lattice(nx, ny, tau, u, delta, 1, storage, bcx, bcy, gx=gx, gy=gy, history_len=hist, layout=layout)
        x.init_fields(rho, ux, uy)
        for b in bodies:
            x.add_markers(b.X, b.Y, b.ds, b.Ubx + 0.01, b.Uby)
        pair.append(x)
    pair[1].tune(1)
    return pair


def same(a, b, last):
    assert np.array_equal(a.field(B.FIELD_POPS), b.field(B.FIELD_POPS))
    for k in range(len(a.body_markers)):
        m, r = a.markers(k), b.markers(k)
        assert all(np.array_equal(m[q], r[q]) for q in m)
        fa, fb = (x.forces(k, x.steps - last, last) for x in (a, b))
        assert np.array_equal(fa[0], fb[0]) and np.array_equal(fa[1], fb[1])


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("nx,ny", [(161, 2051), (64, 64), (300, 1000), (122, 37), (7, 5)])
def test_convective_outlet_with_periodic_rows(nx, ny, storage):
    """The last tile's rows beyond the lattice are its first rows again: only the
    tile that owns them keeps their outlet column."""
    a, b = lattices(nx, ny, storage, W.BCX_CONVECTIVE, W.BCY_PERIODIC)
    for n in (5, 66, 2, 131):
        a.step(n)
        b.step(n)
        same(a, b, 1)


@pytest.mark.parametrize("bcx", [W.BCX_PERIODIC, W.BCX_INOUT, W.BCX_CONVECTIVE])
@pytest.mark.parametrize("storage", STORAGES)
def test_bounce_back_walls_over_many_nodes(storage, bcx):
    """Roundings of the walls' constant that differ once in thousands of nodes."""
    a, b = lattices(2051, 33, storage, bcx, W.BCY_NOSLIP, u=0.06, gx=1e-6 if bcx == W.BCX_PERIODIC else 0.0)
    for n in (70, 131):
        a.step(n)
        b.step(n)
        same(a, b, 1)


@pytest.mark.parametrize("nx,ny,bcx,bcy", [
    (128, 32771, W.BCX_INOUT, W.BCY_FREESLIP),       # 2 nodes per lane for its width
    (2051, 2049, W.BCX_PERIODIC, W.BCY_NOSLIP),      # 4, wrapped columns
    (2050, 2049, W.BCX_PERIODIC, W.BCY_PERIODIC),
    (2049, 2051, W.BCX_CONVECTIVE, W.BCY_PERIODIC),
])
def test_fp32_beyond_l2(nx, ny, bcx, bcy):
    wrap = [W.circle_markers(0.3, ny / 3, 12.0, 37)] if bcx == W.BCX_PERIODIC else []
    a, b = lattices(nx, ny, B.BTDF_F32, bcx, bcy, wrap + [W.circle_markers(nx / 2 + 0.2, ny / 2, 30.0, 94)],
                    gx=1e-6 if bcx == W.BCX_PERIODIC else 0.0)
    before = a.device_bytes()
    for n in (20, 3):
        a.step(n)
        b.step(n)
        same(a, b, n)
    assert a.device_bytes() > before   # the tables of pairs are there


def stable(pair, n):
    """Takes n steps; both sides report a density or force gone astray alike."""
    found = []
    for x in pair:
        x.step(n)
        try:
            x.sync()
            found.append(True)
        except B.BtdfError as e:
            assert e.status == B.BTDF_EUNSTABLE
            found.append(False)
    assert found[0] == found[1]
    return found[0]


def some_bodies(r, nx, ny):
    out = []
    for _ in range(r.choice([0, 1, 1, 2])):
        d = r.uniform(4.0, max(5.0, min(20.0, min(nx, ny) / 3)))
        m = 0.5 * d + 3.2
        if nx > 2 * m + 2 and ny > 2 * m + 2:
            out.append(W.circle_markers(r.uniform(m, nx - 1 - m), r.uniform(m, ny - 1 - m), d, max(6, int(np.pi * d))))
    return out


@pytest.mark.parametrize("seed", range(60))
def test_any_form(seed):
    r = random.Random(seed)
    nx = r.choice([r.randint(4, 70), r.randint(50, 400), r.choice([60, 61, 62, 119, 120, 121, 122, 180, 181, 240, 241, 361])])
    ny = r.choice([r.randint(4, 20), r.randint(15, 120), r.randint(100, 500)])
    bcx, bcy = r.choice([W.BCX_PERIODIC, W.BCX_INOUT, W.BCX_CONVECTIVE]), r.choice([W.BCY_PERIODIC, W.BCY_FREESLIP, W.BCY_NOSLIP])
    u = r.choice([0.05, 0.0, -0.04, 0.1]) if bcx != W.BCX_CONVECTIVE else 0.05
    gx, gy = r.choice([(0.0, 0.0), (0.0, 0.0), (1e-6, 0.0), (1e-6, -2e-6)])
    hist = r.choice([1, 2, 7, 64])
    bodies = some_bodies(r, nx, ny)
    both = lattices(nx, ny, r.choice([B.BTDF_F32, *STORAGES]), bcx, bcy, bodies, r.choice([2, 3, 3, 4, 5]), u, gx, gy,
                    r.uniform(0.7, 1.2), r.choice([B.LAYOUT_ROWS, B.LAYOUT_PLANES]), hist)
    for n in [r.choice([1, 2, 3, 5, 66, 70, 131]) for _ in range(4)]:
        act, dx, factor = r.random(), r.uniform(-0.4, 0.4), r.uniform(0.8, 1.2)
        for x in both:
            if act < 0.15 and bodies:
                x.move_markers(0, bodies[0].X + dx, bodies[0].Y)
            elif act < 0.25 and bcx != W.BCX_PERIODIC:
                x.set_inflow(u * factor)
            elif act < 0.35:
                x.load_state(x.save_state())
            elif act < 0.45 and bodies:
                x.set_marker_velocity(0, np.full(len(bodies[0].X), 0.02 * dx), np.full(len(bodies[0].X), 0.003))
        if not stable(both, n):
            break
        same(*both, min(n, hist))


@pytest.mark.parametrize("seed", range(24))
def test_any_batch(seed):
    r = random.Random(1000 + seed)
    delta, hist, storage = r.choice([2, 3, 4, 5]), r.choice([1, 3, 40]), STORAGES[seed % 3]
    cases = []
    for _ in range(r.randint(2, 6)):
        # half of them without a lattice that takes 4 nodes per lane in FP32
        nx = r.randint(4, 58) if seed % 2 else r.choice([r.randint(4, 400), 121, 61, 241])
        ny = r.randint(4, 150)
        c = W.Case("batch", nx, ny, r.uniform(0.7, 1.2), r.choice([0.05, 0.0, -0.03]), delta,
                   r.choice([W.BCX_PERIODIC, W.BCX_INOUT]), r.choice([W.BCY_PERIODIC, W.BCY_FREESLIP, W.BCY_NOSLIP]),
                   seed=seed, noise=1e-3, gx=r.choice([0.0, 1e-6]))
        c.bodies.extend(some_bodies(r, nx, ny))
        cases.append(c)
    a, b = (B.Batch.from_cases(cases, storage=storage, history_len=hist) for _ in range(2))
    b.tune(1)
    for n in (r.choice([1, 2, 3]), 66, r.choice([2, 5, 33]), 131):
        if not stable((a, b), n):
            break
        for i in range(len(cases)):
            assert np.array_equal(a.field(i, B.FIELD_POPS), b.field(i, B.FIELD_POPS)), (i, n)
        k = min(n, hist)
        for body in range(len(a.bodies)):
            fa, fb = (x.forces(body, x.steps - k, k) for x in (a, b))
            assert np.array_equal(fa[0], fb[0]) and np.array_equal(fa[1], fb[1])


def test_pairs_beside_a_chosen_variant():
    """tune_pairs keeps the variant for the single steps that remain; tune undoes it."""
    body = W.circle_markers(60.3, 30.2, 9.0, 28)
    a, b = lattices(150, 61, B.BTDF_F32, W.BCX_INOUT, W.BCY_FREESLIP, [body])
    a.tune(8)
    before = a.device_bytes()
    a.step(70)
    assert a.device_bytes() == before
    a.tune_pairs()
    a.step(71)
    assert a.device_bytes() > before   # the tables of pairs
    b.step(141)
    same(a, b, 8)
    a.tune(2)
    a.step(5)
    a.tune_pairs(False)
    a.step(2)
    b.step(7)
    same(a, b, 2)


def test_batch_pairs_beside_a_chosen_shape():
    cases = [W.small_cylinder(delta=3), W.small_cylinder(delta=3, seed=9)]
    a, b = (B.Batch.from_cases(cases, history_len=64) for _ in range(2))
    a.tune(2)
    a.tune_pairs()
    b.tune(1)
    for n in (67, 40):
        a.step(n)
        b.step(n)
        for i in range(2):
            assert np.array_equal(a.field(i, B.FIELD_POPS), b.field(i, B.FIELD_POPS))

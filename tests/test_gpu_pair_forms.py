"""Paired steps against single steps in forms that the rule for pairs accepts.
Both sides round alike, so populations, marker results and forces are equal bit
for bit."""
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

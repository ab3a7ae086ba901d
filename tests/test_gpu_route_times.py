"""The kernels that the library chooses by itself are not slower than others it
has for the same work, and right at the edges of their blocks.  Both sides are timed in turn in one process, the lowest
of several runs each; the margins are several times what such runs differ."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1806_09403_gb300 import _build  # noqa: E402
from paper_1806_09403_gb300 import btdf as B  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()


def lattice(nx, ny, storage, bcx=W.BCX_INOUT, bcy=W.BCY_FREESLIP):
    lat = B.Lattice(nx, ny, 0.6, 0.05, 3, 1, storage, bcx, bcy, stream=torch.cuda.current_stream().cuda_stream)
    one = np.ones((ny, nx))
    lat.init_fields(one, 0.05 * one, 0.0 * one)
    return lat


def lowest(runs, rounds=6):
    """Lowest time of each callable in us, timed in turn."""
    best = [float("inf")] * len(runs)
    for r in range(rounds + 1):
        for k, f in enumerate(runs):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            f()
            b.record()
            b.synchronize()
            if r:
                best[k] = min(best[k], 1e3 * a.elapsed_time(b))
    return best


def test_two_node_register_kernel_streams_like_the_four_node_one():
    """FP32 beyond L2: the single step of lattices below 2^23 nodes (variant 2)
    against variant 1 (equal within 1% where the address of its stores is formed
    late, 13% slower where it is not)."""
    lats = [lattice(2048, 2048, B.BTDF_F32) for _ in range(2)]
    for x, v in zip(lats, (2, 1)):
        x.tune(v)
    two, four = lowest([lambda x=x: x.step(64) for x in lats])
    assert two < 1.06 * four, (two, four)


@pytest.mark.parametrize("nx,ny,storage,bcx,single", [
    # the outlet column's nine loads on one path (12% slower than single steps one by one)
    (160, 80, B.BTDF_F32, W.BCX_CONVECTIVE, 2),
    (320, 160, B.BTDF_F32, W.BCX_CONVECTIVE, 2),
    # strips of pairs that leave many columns unused (10 to 40% slower than single steps)
    (124, 16912, B.BTDF_F16DEV, W.BCX_INOUT, 11),
    (128, 16384, B.BTDF_BF16DEV, W.BCX_PERIODIC, 11),
    (250, 8388, B.BTDF_F16DEV, W.BCX_INOUT, 11),
    (124, 2114, B.BTDF_F32, W.BCX_INOUT, 2),
    (121, 16384, B.BTDF_F32, W.BCX_INOUT, 2),
    (128, 65536, B.BTDF_F32, W.BCX_INOUT, 11),
])
def test_automatic_steps_are_not_slower_than_single_ones(nx, ny, storage, bcx, single):
    lats = [lattice(nx, ny, storage, bcx) for _ in range(2)]
    lats[1].tune(single)
    steps = 512 if nx * ny < 1 << 22 else 64
    auto, one = lowest([lambda x=x: x.step(steps) for x in lats])
    assert auto < 1.04 * one, (auto, one)


def test_reading_a_narrow_lattice():
    """Lattices 4 nodes wide are padded to 32 columns, so reading one costs some
    three times what a wide one of as many nodes does (17 times where every row has
    blocks of its own)."""
    lats = [lattice(4, 1 << 20, B.BTDF_F32), lattice(2048, 2048, B.BTDF_F32)]
    out = torch.empty(9 << 22, device="cuda")
    for x in lats:
        x.step(2)
    narrow, wide = lowest([lambda x=x: x.field_to_device(B.FIELD_POPS, out.data_ptr()) for x in lats])
    assert narrow < 8 * wide, (narrow, wide)


@pytest.mark.parametrize("storage,half_ulp", [(B.BTDF_F32, 2.0 ** -24), (B.BTDF_F16DEV, 2.0 ** -12),
                                              (B.BTDF_BF16DEV, 2.0 ** -9)])
@pytest.mark.parametrize("nx,ny", [(4, 4), (5, 61), (16, 65), (255, 7), (256, 4), (257, 9)])
def test_reading_fields_at_block_edges(nx, ny, storage, half_ulp):
    """Rows that end within a block of the read-out.  A new lattice's moments are
    its initial fields up to the rounding of nine stored deviations of at most
    0.1, and of the read-out's own sums in FP32."""
    lat = lattice(nx, ny, storage)
    rng = np.random.default_rng(nx * ny)
    rho, ux, uy = (c + rng.uniform(-0.02, 0.02, (ny, nx)) for c in (1.0, 0.05, 0.0))
    lat.init_fields(rho, ux, uy)
    tol = 2 * 9 * 0.1 * half_ulp + 1e-6
    for want, kind in ((rho, B.FIELD_RHO), (ux, B.FIELD_UX), (uy, B.FIELD_UY)):
        assert np.abs(lat.field(kind) - want).max() < tol
    pops = lat.field(B.FIELD_POPS)
    assert np.abs(pops.sum(0) - rho).max() < tol

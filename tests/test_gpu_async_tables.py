"""The step call that builds the tables of the paired steps: it returns while
earlier work of its stream is still running, and it works while a stream that has
nothing to do with it is being captured."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1806_09403_gb300 import _build  # noqa: E402
from paper_1806_09403_gb300 import btdf as B  # noqa: E402

BUSY_CYCLES = 1_000_000_000   # half a second of device time at 2 GHz


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()


def case():
    c = W.Case("tables", 200, 90, 0.6, 0.04, 3, W.BCX_INOUT, W.BCY_FREESLIP, seed=6, noise=1e-3)
    c.bodies.append(W.circle_markers(60.3, 40.2, 12.0, 37))
    return c


def cylinders(nx, ny, count):
    c = W.Case("many", nx, ny, 0.6, 0.04, 3, W.BCX_INOUT, W.BCY_FREESLIP)
    cols = max(1, round((count * nx / ny) ** 0.5))
    rows = -(-count // cols)
    for k in range(count):
        c.bodies.append(W.circle_markers((k % cols + 0.5) * nx / cols, (k // cols + 0.5) * ny / rows, 40.0, 126))
    return c


def single(stream):
    x = B.Lattice.from_case(case(), stream=stream.cuda_stream)
    return x, lambda: [x.field(B.FIELD_POPS)]


def many(stream):   # tables of half a megabyte: small copies of pageable memory
    x = B.Lattice.from_case(cylinders(1200, 800, 60), stream=stream.cuda_stream)
    return x, lambda: [x.field(B.FIELD_POPS)]


def crowd(stream):   # tables beyond a megabyte: page-locked memory
    x = B.Lattice.from_case(cylinders(1200, 800, 130), stream=stream.cuda_stream)
    return x, lambda: [x.field(B.FIELD_POPS)]


def batch(stream):
    x = B.Batch.from_cases([case(), case()], stream=stream.cuda_stream)
    return x, lambda: [x.field(i, B.FIELD_POPS) for i in range(2)]


def loaded(make, *calls):
    """The result of the same calls, which also loads every kernel they use."""
    x, fields = make(torch.cuda.Stream())
    for n in calls:
        x.step(n)
    return fields()


@pytest.mark.parametrize("make", [single, many, crowd, batch])
def test_building_the_tables_does_not_wait_for_the_stream(make):
    want = loaded(make, 40, 60)
    s = torch.cuda.Stream()
    x, fields = make(s)
    done = torch.cuda.Event()
    for n in (40, 60):
        with torch.cuda.stream(s):
            torch.cuda._sleep(BUSY_CYCLES)
            done.record(s)
        x.step(n)
        assert not done.query(), n
        s.synchronize()
    assert all(np.array_equal(a, b) for a, b in zip(fields(), want))


@pytest.mark.parametrize("make,n", [(single, 63), (batch, 31)])   # one step short of the internal graphs
def test_building_the_tables_while_another_stream_is_captured(make, n):
    want = loaded(make, 1, n)
    x, fields = make(torch.cuda.Stream())
    x.step(1)
    x.sync()
    t = torch.ones(16, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream(), capture_error_mode="global"):
        u = t + 1.0
        x.step(n)
    g.replay()
    assert all(np.array_equal(a, b) for a, b in zip(fields(), want))
    assert float(u.sum()) == 32.0


@pytest.mark.parametrize("storage,nx,ny,bodies,steps,built_then", [
    (B.BTDF_F16DEV, 4096, 1024, 1, 40, True),     # one body's tables pay after 9 steps
    (B.BTDF_F32, 2048, 2048, 1, 10, True),        # after 3
    (B.BTDF_F32, 2048, 2048, 100, 33, False),     # a hundred bodies' after 107
    (B.BTDF_F32, 2048, 2048, 100, 110, True),
])
def test_tables_are_built_once_the_steps_pay_for_them(storage, nx, ny, bodies, steps, built_then):
    x = B.Lattice.from_case(cylinders(nx, ny, bodies), storage=storage, history_len=256)
    before = x.device_bytes()
    x.step(steps)
    x.sync()
    assert (x.device_bytes() > before) == built_then


def test_short_first_call_of_a_batch_builds_no_tables():
    """Three steps of a new batch, against launch shape 3, which has no tables
    (four times its time with them)."""
    import time
    cases = [cylinders(256 + 16 * i, 160, 2) for i in range(24)]
    best = {0: 1e9, 3: 1e9}
    for _ in range(4):
        for shape in best:
            x = B.Batch.from_cases(cases, history_len=64)
            x.tune(shape)
            x.sync()
            t = time.perf_counter()
            x.step(3)
            x.sync()
            best[shape] = min(best[shape], time.perf_counter() - t)
            x.close()
    assert best[0] < 1.6 * best[3], best

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


def single(stream):
    x = B.Lattice.from_case(case(), stream=stream.cuda_stream)
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


@pytest.mark.parametrize("make", [single, batch])
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

"""Step calls that the caller captures into a CUDA graph of its own: a call of an
even number of steps ends in the population buffer it began with, however its
steps are grouped, so every replay goes on from the one before."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1806_09403_gb300 import _build  # noqa: E402
from paper_1806_09403_gb300 import btdf as B  # noqa: E402

LEAD = 70   # enough steps for the tables of the pairs to be there


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()


def case(bcx, bodies):
    c = W.Case("capture", 150, 61, 0.6, 0.04, 3, bcx, W.BCY_FREESLIP, seed=5, noise=1e-3)
    if bodies:
        c.bodies.append(W.circle_markers(60.3, 30.2, 9.0, 28))
    return c


def replayed(x, stream, n, replays):
    """Captures x.step(n) on the stream of x and replays it."""
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        x.step(n)
    with torch.cuda.stream(stream):
        for _ in range(replays):
            g.replay()
    stream.synchronize()
    return g


@pytest.mark.parametrize("n", [2, 3, 4, 6])
@pytest.mark.parametrize("bodies", [False, True])
@pytest.mark.parametrize("bcx", [W.BCX_INOUT, W.BCX_CONVECTIVE])
def test_replays_advance(n, bodies, bcx):
    s = torch.cuda.Stream()
    c = case(bcx, bodies)
    a = B.Lattice.from_case(c, stream=s.cuda_stream)
    b = B.Lattice.from_case(c)
    replays = 3 if n % 2 == 0 else 1   # an odd count ends in the other buffer
    a.step(LEAD)
    b.step(LEAD + replays * n)
    g = replayed(a, s, n, replays)   # noqa: F841  (the graph outlives its replays)
    assert np.array_equal(a.field(B.FIELD_POPS), b.field(B.FIELD_POPS))


@pytest.mark.parametrize("n", [2, 3, 4, 6])
@pytest.mark.parametrize("bodies", [False, True])
def test_batch_replays_advance(n, bodies):
    s = torch.cuda.Stream()
    cases = [case(W.BCX_INOUT, bodies), case(W.BCX_PERIODIC, False)]
    a = B.Batch.from_cases(cases, stream=s.cuda_stream)
    b = B.Batch.from_cases(cases)
    replays = 3 if n % 2 == 0 else 1
    a.step(LEAD)
    b.step(LEAD + replays * n)
    g = replayed(a, s, n, replays)   # noqa: F841
    for i in range(len(cases)):
        assert np.array_equal(a.field(i, B.FIELD_POPS), b.field(i, B.FIELD_POPS))

"""Advances captured by the caller: each replay goes on from the state that the last
one left, so a captured advance takes a form that ends in the row it began in."""
import numpy as np
import pytest

from helpers import spec_for, state_for
from paper_1705_03162_gb300 import build as B
from paper_1705_03162_gb300 import swept as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()
    S.load_library()


def _classic(spec, u0, dtype, steps):
    with S.Problem(spec, u0, dtype) as q:
        q.advance(steps, "classic")
        return q.read()


@pytest.mark.parametrize("eq,N,steps", [("ks", (1 << 22) + 3, 4), ("ks", 1 << 22, 21), ("heat", (1 << 22) + 5, 30)])
def test_captured_tiled_advance_replays(eq, N, steps):
    """FP32 grids beyond the chip: the default advance is a launch per some ten
    levels from row to row, an odd number of them for some step counts."""
    torch = pytest.importorskip("torch")
    spec = spec_for(eq, "periodic", N)
    u0 = state_for(spec, np.float32)
    stream = torch.cuda.Stream()
    with S.Problem(spec, u0, "f32", stream=stream) as p:
        p.advance(2, "swept")
        p.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            p.advance(steps, "swept")
        with torch.cuda.stream(stream):
            for _ in range(3):
                g.replay()
        assert np.array_equal(p.read(), _classic(spec, u0, "f32", 2 + 3 * steps))

"""Advances captured by the caller: each replay goes on from the state that the last
one left, so a captured advance takes a form that ends in the row it began in."""
import threading

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


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_captured_batch_advance_replays(dtype):
    """A batch that runs on chip by default (from row to row), captured."""
    torch = pytest.importorskip("torch")
    specs = [spec_for("ks", "periodic", 3001), spec_for("heat", "periodic", 2000), spec_for("heat", "reflective", 777)]
    u0 = [state_for(s, np.float64 if dtype == "f64" else np.float32, seed=i) for i, s in enumerate(specs)]
    steps = [9, 10, 12]
    stream = torch.cuda.Stream()
    probs = [S.Problem(s, u, dtype, stream=stream) for s, u in zip(specs, u0)]
    with S.Batch(stream) as b:
        b.advance(probs, [2, 2, 2])
        b.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream, capture_error_mode="relaxed"):
            b.advance_ex(probs, steps, ["swept"] * 3)
        with torch.cuda.stream(stream):
            for _ in range(3):
                g.replay()
        b.synchronize()
        for s, u, st, p in zip(specs, u0, steps, probs):
            assert np.array_equal(p.read(), _classic(s, u, dtype, 2 + 3 * st)), (s.eq, s.bc)
            p.close()


@pytest.mark.parametrize("eq,bc,N,dtype", [("heat", "periodic", 1024, "f64"), ("ks", "periodic", 2048, "f32"),
                                           ("euler", "dirichlet", 300, "f64")])
def test_first_advance_beside_another_threads_capture(eq, bc, N, dtype):
    """A problem's first default advance (it allocates its halo words) while
    another thread captures its own stream: both go through."""
    torch = pytest.importorskip("torch")
    spec = spec_for(eq, bc, N)
    u0 = state_for(spec, np.float64 if dtype == "f64" else np.float32)
    begun, done, out = threading.Event(), threading.Event(), []

    def capture():
        try:
            x = torch.zeros(8, device="cuda")
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=torch.cuda.Stream()):   # the default: global mode
                x += 1
                begun.set()
                done.wait(30)
            g.replay()
            torch.cuda.synchronize()
            out.append(float(x[0]))
        finally:
            begun.set()

    with S.Problem(spec, u0, dtype, stream=torch.cuda.Stream()) as p:
        th = threading.Thread(target=capture)
        th.start()
        try:
            assert begun.wait(30)
            p.advance(20, "swept")
        finally:
            done.set()
            th.join()
        assert out == [1.0]
        assert p.kernel_launches() == 1
        assert np.array_equal(p.read(), _classic(spec, u0, dtype, 20))

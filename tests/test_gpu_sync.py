"""What a wait for a problem's stream costs: its own stream's work, and no more."""
import time

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


@pytest.mark.parametrize("eq,bc,N,dtype", [("heat", "periodic", 1024, "f64"), ("ks", "periodic", 5001, "f32"),
                                           ("euler", "dirichlet", 300, "f64")])
def test_default_advance_does_not_wait_for_other_streams(eq, bc, N, dtype):
    """synchronize and a read to host memory after a default (on-chip) advance
    return while the legacy default stream is still busy (about 0.5 s)."""
    torch = pytest.importorskip("torch")
    spec = spec_for(eq, bc, N)
    u0 = state_for(spec, np.float64 if dtype == "f64" else np.float32)
    with S.Problem(spec, u0, dtype, stream=torch.cuda.Stream()) as p, S.Problem(spec, u0, dtype) as q:
        for _ in range(2):
            p.advance(10, "swept")
            p.read()
        q.advance(30, "classic")
        want = q.read()
        torch.cuda.synchronize()
        busy = torch.cuda.Event()
        torch.cuda._sleep(1_000_000_000)
        busy.record()
        t0 = time.perf_counter()
        p.advance(10, "swept")
        p.synchronize()
        got = p.read()
        took = time.perf_counter() - t0
        still = not busy.query()
        torch.cuda.synchronize()
        assert still and took < 0.2, took
        assert np.array_equal(got, want)


def test_persistent_advance_does_not_wait_for_other_streams():
    """The same for a launch whose status word is device memory."""
    torch = pytest.importorskip("torch")
    spec = spec_for("ks", "periodic", 4096)
    u0 = state_for(spec)
    with S.Problem(spec, u0, stream=torch.cuda.Stream()) as p:
        for _ in range(2):
            p.advance(10, "swept", 256, "persistent")
            p.read()
        torch.cuda.synchronize()
        busy = torch.cuda.Event()
        torch.cuda._sleep(1_000_000_000)
        busy.record()
        p.advance(10, "swept", 256, "persistent")
        p.synchronize()
        still = not busy.query()
        torch.cuda.synchronize()
        assert still


def test_creating_and_closing_problems_costs_no_pinned_memory():
    """A problem's life (create, a short default advance, read, close) takes no longer
    than twice that of a problem that runs per-phase launches, which have no words:
    a pinned allocation and its release alone take longer than the rest."""
    spec = spec_for("heat", "periodic", 1024)
    u0 = state_for(spec)

    def life(n, launch):
        took = []
        for _ in range(60):
            t0 = time.perf_counter()
            with S.Problem(spec, u0) as p:
                p.advance(10, "swept", n, launch)
                p.read()
            took.append(time.perf_counter() - t0)
        return float(np.median(took[20:]))

    life(0, "auto")
    assert life(0, "auto") < 2 * life(128, "per_phase")

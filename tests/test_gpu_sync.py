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

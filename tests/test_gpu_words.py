"""The published words of a single on-chip advance: sequence numbers that start over,
waits that run out, in every kernel that polls them, and which Euler grids have them."""
import time

import numpy as np
import pytest

from helpers import spec_for, state_for
from paper_1705_03162_gb300 import build as B
from paper_1705_03162_gb300 import swept as S

pytestmark = pytest.mark.gpu

CASES = [("heat", "periodic", 4099, "f64"), ("ks", "periodic", 3001, "f32"), ("heat", "reflective", 1500, "f32"),
         ("euler", "dirichlet", 1001, "f64"), ("euler", "periodic", 20001, "f64")]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()
    S.load_library()


def _case(eq, bc, N, dtype):
    spec = spec_for(eq, bc, N)
    return spec, state_for(spec, np.float64 if dtype == "f64" else np.float32)


def _classic(spec, u0, dtype, steps):
    with S.Problem(spec, u0, dtype) as q:
        q.advance(steps, "classic")
        return q.read()


@pytest.mark.parametrize("eq,bc,N,dtype", CASES)
def test_sequence_numbers_start_over(eq, bc, N, dtype):
    """An advance that would pass 2^31 starts over on cleared words; the one before
    it, close to 2^31, and those after it give the same bits."""
    spec, u0 = _case(eq, bc, N, dtype)
    with S.Problem(spec, u0, dtype) as p:
        with pytest.raises(S.SweptError) as e:
            p.debug_sequence(1 << 30)
        assert e.value.status == S.EINVAL
        p.advance(150, "swept")
        p.debug_sequence((1 << 31) - 200)
        p.advance(150, "swept")       # fits below 2^31
        p.debug_sequence((1 << 31) - 1)
        for _ in range(3):
            p.advance(150, "swept")   # the first of these starts over
        assert p.kernel_launches() == 5
        assert np.array_equal(p.read(), _classic(spec, u0, dtype, 750))


@pytest.mark.parametrize("eq,bc,N,dtype", CASES)
def test_withheld_words_time_out_and_recover(eq, bc, N, dtype):
    """Advances long enough for an exchange (small FP32 grids: after some hundred levels)."""
    spec, u0 = _case(eq, bc, N, dtype)
    with S.Problem(spec, u0, dtype) as p:
        p.debug_withhold_flags(True, wait_limit_ns=100_000_000)
        t0 = time.perf_counter()
        p.advance(2000, "swept")
        with pytest.raises(S.SweptError) as e:
            p.synchronize()
        assert e.value.status == S.ETIMEOUT
        assert time.perf_counter() - t0 < 5
        p.debug_withhold_flags(False)
        p.write(u0)
        p.advance(2000, "swept")
        assert np.array_equal(p.read(), _classic(spec, u0, dtype, 2000))


@pytest.mark.parametrize("bc,N,on_chip", [("dirichlet", 57001, True), ("dirichlet", 57301, False),
                                          ("dirichlet", 131072, False), ("periodic", 131072, True)])
def test_euler_form_by_boundary(bc, N, on_chip):
    """A Dirichlet tube's default advance leaves the chip where the dataflow launch
    becomes the faster form (a problem without on-chip words has no sequence)."""
    spec, u0 = _case("euler", bc, N, "f64")
    with S.Problem(spec, u0, "f64") as p:
        p.advance(12, "swept")
        if on_chip:
            p.debug_sequence(1 << 20)
        else:
            with pytest.raises(S.SweptError) as e:
                p.debug_sequence(1 << 20)
            assert e.value.status == S.EINVAL
        p.advance(5, "swept")
        assert np.array_equal(p.read(), _classic(spec, u0, "f64", 17))

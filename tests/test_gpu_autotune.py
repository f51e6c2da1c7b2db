"""What the autotuners keep: after tuning, SWP_SCHEME_AUTO advances and default
batches are no slower than before, because the default launch is measured too."""

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


def _launches(p, steps, scheme):
    k0 = p.kernel_launches()
    p.advance(steps, scheme)
    return p.kernel_launches() - k0


# sizes at which the default launch is on chip, several times as fast as any width
@pytest.mark.parametrize("eq,bc,N,dtype", [("heat", "periodic", 1016, "f64"), ("ks", "periodic", 4104, "f64"),
                                           ("heat", "reflective", 131064, "f32"), ("ks", "periodic", 65544, "f32"),
                                           ("euler", "dirichlet", 3999, "f64")])
@pytest.mark.parametrize("width_only", [False, True])
def test_tuning_keeps_the_default_launch_where_it_is_faster(eq, bc, N, dtype, width_only):
    torch = pytest.importorskip("torch")
    spec = spec_for(eq, bc, N + (16 if width_only else 0))   # a key of its own
    u0 = state_for(spec, np.float64 if dtype == "f64" else np.float32)
    if width_only:
        n = S.autotune_width(spec, u0, count=4, steps=300, dtype=dtype)
        assert n == S.tuned_width(spec, dtype) and n >= 32
    else:
        assert S.autotune(spec, u0, count=4, steps=300, dtype=dtype) == S.tuned(spec, dtype)
    with S.Problem(spec, u0, dtype) as p, S.Problem(spec, u0, dtype) as q:
        assert _launches(p, 300, "auto") == _launches(p, 300, "swept") == 1
        q.advance(600, "classic")
        assert np.array_equal(p.read(), q.read())
    if eq != "euler" and dtype == "f32":
        stream = torch.cuda.Stream()
        ps = [S.Problem(spec, u0, dtype, stream=stream) for _ in range(4)]
        with S.Batch(stream) as b:
            b.advance_ex(ps, [50] * 4)
            assert b.debug_form() == (4, 0)
            b.synchronize()
        for p in ps:
            p.close()


def test_failed_tuning_keeps_the_earlier_choice():
    """Tuning that cannot create its problems (the memory budget) returns an error
    and leaves what was tuned before."""
    spec = spec_for("heat", "periodic", 1040)
    u0 = state_for(spec)
    n = S.autotune_width(spec, u0, count=2, steps=50)
    S.set_memory_budget(1)
    try:
        with pytest.raises(S.SweptError):
            S.autotune_width(spec, u0, count=2, steps=50)
    finally:
        S.set_memory_budget(0)
    assert S.tuned_width(spec) == n

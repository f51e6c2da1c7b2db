"""Which form a batch of heat and KS problems takes (on chip, or the table form with
which node widths), and that each gives the classic scheme's bits."""
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


KINDS = [("heat", "periodic"), ("ks", "periodic"), ("heat", "reflective")]


class Set:
    """Problems of these sizes, kinds in turn, on a stream of their own."""

    def __init__(self, dtype, sizes, steps, kinds=KINDS):
        torch = pytest.importorskip("torch")
        self.dtype, self.stream = dtype, torch.cuda.Stream()
        self.specs = [spec_for(*kinds[i % len(kinds)], n) for i, n in enumerate(sizes)]
        npdt = np.float64 if dtype == "f64" else np.float32
        self.u0 = [state_for(s, npdt, seed=i) for i, s in enumerate(self.specs)]
        self.steps = [steps + (7 * i) % 23 for i in range(len(sizes))]
        self.probs = [S.Problem(s, u, dtype, stream=self.stream) for s, u in zip(self.specs, self.u0)]

    def check(self, times):
        """Every state is `times` advances of the classic scheme; ends the set."""
        for s, u, st, p in zip(self.specs, self.u0, self.steps, self.probs):
            with S.Problem(s, u, self.dtype) as q:
                q.advance(times * st, "classic")
                assert np.array_equal(p.read(), q.read()), (s.eq, s.bc, s.n_points, st)
            p.close()


def _nodes(specs, widths):
    return sum(s.n_points // w for s, w in zip(specs, widths))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("sizes", [[1031, 2503, 4099, 3000], [15001 + 31 * i for i in range(12)]])
def test_given_widths_hold_in_the_table_form(dtype, sizes):
    """Odd sizes with widths that leave remainders: with launch "persistent" and
    with a given block size the batch runs exactly these nodes."""
    s = Set(dtype, sizes, 150)
    step = 8
    widths = [step * (9 + 5 * i) for i in range(len(sizes))]
    assert any(n % w for n, w in zip(sizes, widths))
    with S.Batch(s.stream) as b:
        b.advance_ex(s.probs, s.steps, ["swept"] * len(sizes), widths, launch="persistent")
        assert b.debug_form() == (0, _nodes(s.specs, widths))
        b.advance_ex(s.probs, s.steps, ["swept"] * len(sizes), widths, threads=64, launch="graph")
        assert b.debug_form() == (0, _nodes(s.specs, widths))
        b.synchronize()
    s.check(2)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_tune_width_times_the_widths_it_returns(dtype):
    """The trials run the table form with the candidate's widths (the last one's
    nodes are those of the last advance), in groups that run on chip by default."""
    s = Set(dtype, [2503, 4099, 3001], 120)
    candidates = (64, 1000, 256)
    with S.Batch(s.stream) as b:
        widths, best, ms = b.tune_width(s.probs, s.steps, candidates)
        last = [S.fit_width(x.eq, x.n_points, candidates[-1]) for x in s.specs]
        assert b.debug_form() == (0, _nodes(s.specs, last))
        assert widths == [S.fit_width(x.eq, x.n_points, candidates[best]) for x in s.specs]
        b.advance_ex(s.probs, s.steps, ["swept"] * 3, widths, launch="persistent")
        assert b.debug_form() == (0, _nodes(s.specs, widths))
        b.advance(s.probs, s.steps)
        assert b.debug_form() == (3, 0)
        b.synchronize()
    s.check(2)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("launch", ["auto", "graph"])
def test_refused_on_chip_launch_takes_the_table_form(dtype, launch):
    """A device that cannot hold the cooperative launch: the same advance in the
    table form, also later without asking again, and on chip once it can."""
    s = Set(dtype, [1031, 2503, 4099], 100)
    with S.Batch(s.stream) as b:
        b.debug_refuse(True)
        for _ in range(2):
            b.advance_ex(s.probs, s.steps, ["swept"] * 3, launch=launch)
            on_chip, nodes = b.debug_form()
            assert on_chip == 0 and nodes >= 6
        b.debug_refuse(False)
        b.advance_ex(s.probs, s.steps, ["swept"] * 3, launch=launch)
        assert b.debug_form() == (3, 0)
        b.synchronize()
        assert b.kernel_launches() == 3
    s.check(3)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("launch", ["auto", "graph"])
def test_withheld_words_of_a_batch_time_out_and_recover(dtype, launch):
    """Problems of several tiles among which one has its words withheld: every
    wait of the launch gives up within the limit (blocks whose tiles are still
    unclaimed leave too), synchronize reports it, and the batch runs again once
    the states are rewritten."""
    sizes = [1031, 4099, 2503, 30, 3000] if dtype == "f64" else [15000] * 90 + [4099, 30]
    s = Set(dtype, sizes, 100)
    schemes = ["swept"] * len(sizes)
    with S.Batch(s.stream) as b:
        b.advance_ex(s.probs, s.steps, schemes, launch=launch)
        assert b.debug_form() == (len(sizes), 0)
        b.synchronize()
        s.probs[1].debug_withhold_flags(True, wait_limit_ns=100_000_000)
        for _ in range(2):
            t0 = time.perf_counter()
            b.advance_ex(s.probs, s.steps, schemes, launch=launch)
            assert b.debug_form() == (len(sizes), 0)
            with pytest.raises(S.SweptError) as e:
                b.synchronize()
            assert e.value.status == S.ETIMEOUT
            assert time.perf_counter() - t0 < 5
        s.probs[1].debug_withhold_flags(False)
        for p, u in zip(s.probs, s.u0):
            p.write(u)
        for _ in range(2):
            b.advance_ex(s.probs, s.steps, schemes, launch=launch)
        b.synchronize()
    s.check(2)

"""The batched on-chip tiles of both lengths and precisions, on problems of one tile
(its halos are its own points), two and many, with the tile length asserted: a batch
whose tile length is chosen differently fails here rather than test something else."""
import pytest

from helpers import spec_for
from paper_1705_03162_gb300 import build as B
from paper_1705_03162_gb300 import swept as S
from test_gpu_batch_forms import KINDS, Set

pytestmark = pytest.mark.gpu

# points that a tile owns: slots less the halos on both sides
SHORT = {"f64": 88, "f32": 832}
LONG = {"f64": 216, "f32": 1856}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()
    S.load_library()


def _tiles(sizes, own):
    return sum(-(-n // own) for n in sizes)


def _edges(own):
    """Sizes around one and two tiles, and the smallest that run swept."""
    return [16, 21, own - 1, own, own + 1, 2 * own - 1, 2 * own, 2 * own + 1, 3 * own + 5]


def _each_kind(sizes):
    return [n for n in sizes for _ in KINDS]


# (sizes, tile length): FP64 takes the short tiles up to about 53 k points in all, the
# long ones up to about 80 k; FP32 the long ones from 2.5 tiles per place of the chip
CASES = [
    ("f64", _each_kind(_edges(88)), SHORT),
    ("f64", _each_kind(_edges(216)) + [2001 + 7 * i for i in range(16)], SHORT),
    ("f64", _each_kind(_edges(88) + _edges(216)) + [3001 + 11 * i for i in range(16)], LONG),
    ("f64", [9001], SHORT),
    ("f64", [9001 + 500 * i for i in range(5)], SHORT),
    ("f64", [11001 + 1000 * i for i in range(5)], LONG),
    ("f64", [70001], LONG),
    ("f32", _each_kind(_edges(832)) + [100003], SHORT),
    ("f32", _each_kind(_edges(1856)) + [30011] * 100, LONG),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("steps", [1, 64])
def test_tiles(case, steps):
    """Advances of one step to several exchanges (7 i mod 23 more for problem i),
    twice through a cached graph per row and once as a plain launch."""
    dtype, sizes, own = CASES[case]
    s = Set(dtype, sizes, steps)
    n = len(sizes)
    with S.Batch(s.stream) as b:
        for launch in ("graph", "graph", "graph", "auto"):
            b.advance_ex(s.probs, s.steps, ["swept"] * n, launch=launch)
            assert b.debug_form() == (n, 0) and b.debug_tiles() == _tiles(sizes, own[dtype])
        b.synchronize()
    s.check(4)


@pytest.mark.parametrize("dtype,sizes", [("f32", [1150003, 2503, 4099]), ("f64", [1000003, 30011, 40009, 50021])])
def test_long_problem_sends_the_group_to_the_table_form(dtype, sizes):
    """FP32: more tiles than the launch has blocks; FP64: a problem that is most of
    the batch's time.  The given widths hold."""
    s = Set(dtype, sizes, 20)
    widths = [S.fit_width(x.eq, x.n_points, 700) for x in s.specs]
    with S.Batch(s.stream) as b:
        b.advance_ex(s.probs, s.steps, ["swept"] * len(sizes), widths)
        assert b.debug_form() == (0, sum(x.n_points // w for x, w in zip(s.specs, widths)))
        b.synchronize()
    s.check(1)


def test_fp64_groups_by_size():
    """Below and above the size up to which an FP64 group runs on chip."""
    for sizes, on_chip in (([70001], True), ([90001], False)):
        s = Set("f64", sizes, 10)
        with S.Batch(s.stream) as b:
            b.advance(s.probs, s.steps)
            assert (b.debug_form()[0] > 0) == on_chip
            b.synchronize()
        s.check(1)


def test_smallest_problems_are_swept():
    """The sizes above that run on chip are no classic items (two nodes of 4 rad)."""
    assert all(S.fit_width(spec_for(eq, bc, 16).eq, 16, 8) > 0 for eq, bc in KINDS)

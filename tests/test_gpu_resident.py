"""The resident form (the default launch of heat and KS where the grid fits the
chip, and tiles of the same kind for larger FP32 grids): blocks exchange halos
through published words, so every point must equal the CPU oracle's bit for bit
whatever the tile shape, the number of exchanges and the boundary, on repeated
advances, on concurrent streams and under capture; a wait that cannot succeed
ends in SWP_ETIMEOUT."""
import time

import numpy as np
import pytest

import oracle as O
from helpers import oprob, spec_for, state_for
from paper_1705_03162_gb300 import build as B
from paper_1705_03162_gb300 import swept as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()
    S.load_library()


def _np(dtype):
    return np.float64 if dtype == "f64" else np.float32


def _oracle(spec, u0, steps):
    ref = np.ascontiguousarray(u0.copy())
    O.classic(oprob(spec), ref, steps)
    return ref


# sizes around the plan's choices: few blocks, halos over several blocks, over
# more than one period, blocks of unequal length, one and several warps per SM
# sub-partition, blocks whose ends alone are published
SIZES = (64, 65, 97, 255, 1021, 2433, 4099, 10007, 19457, 50001, 65537)


@pytest.mark.parametrize("eq,bc", [("heat", "periodic"), ("heat", "reflective"), ("ks", "periodic")])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("N", SIZES)
def test_default_launch_any_size(eq, bc, dtype, N):
    """Advances shorter than an exchange, an odd number of levels, and several
    exchanges with a remainder, one after the other on the same problem."""
    spec = spec_for(eq, bc, N)
    u0 = state_for(spec, _np(dtype), seed=N)
    ref = u0.copy()
    with S.Problem(spec, u0, dtype) as p:
        for steps in (1, 7, 400 if N < 5000 else 151):
            k0 = p.kernel_launches()
            p.advance(steps, "swept")
            assert p.kernel_launches() - k0 == 1
            O.classic(oprob(spec), ref, steps)
            assert np.array_equal(p.read(), ref), steps


@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
@pytest.mark.parametrize("N", [32, 33, 61, 150, 1021, 4099, 16400, 20001])
def test_default_launch_euler_any_size(bc, N):
    """Tiles with ghost cells on one or both sides, halos over several blocks and
    more than one period, one and several rows of cells per sub-partition."""
    spec = spec_for("euler", bc, N)
    u0 = state_for(spec, seed=N)
    ref = u0.copy()
    with S.Problem(spec, u0) as p:
        for steps in (1, 5, 120 if N < 5000 else 40):
            k0 = p.kernel_launches()
            p.advance(steps, "swept")
            assert p.kernel_launches() - k0 == 1
            O.classic(oprob(spec), ref, steps)
            assert np.array_equal(p.read(), ref), steps


@pytest.mark.parametrize("eq,bc,N,dtype,steps", [
    ("euler", "periodic", 200003, "f64", 30), ("euler", "dirichlet", 300001, "f64", 30),
    ("heat", "reflective", (1 << 17) + 1, "f64", 90), ("heat", "periodic", 400009, "f64", 60),
    ("heat", "periodic", (1 << 20) + 7, "f64", 70), ("heat", "reflective", 700001, "f32", 333),
    ("ks", "periodic", 300007, "f32", 120), ("ks", "periodic", 2097152, "f32", 100),
    ("ks", "periodic", (1 << 22) + 3, "f32", 90), ("heat", "reflective", (1 << 22) + 9, "f32", 401)])
def test_default_launch_large_equals_classic(eq, bc, N, dtype, steps):
    spec = spec_for(eq, bc, N)
    u0 = state_for(spec, _np(dtype), seed=3)
    with S.Problem(spec, u0, dtype) as p, S.Problem(spec, u0, dtype) as q:
        p.advance(steps, "swept")
        q.advance(steps, "classic")
        assert np.array_equal(p.read(), q.read())


def test_concurrent_streams():
    """Several problems advancing at once on streams of their own, many short
    advances each: every launch needs all its blocks resident."""
    torch = pytest.importorskip("torch")
    cases = [("heat", "periodic", 4099, "f64"), ("ks", "periodic", 20011, "f32"), ("heat", "reflective", 1500, "f32"),
             ("ks", "periodic", 1031, "f64")]
    streams = [torch.cuda.Stream() for _ in cases]
    specs = [spec_for(eq, bc, N) for eq, bc, N, _ in cases]
    u0 = [state_for(s, _np(c[3]), seed=5) for s, c in zip(specs, cases)]
    probs = [S.Problem(s, u, c[3], stream=st) for s, u, c, st in zip(specs, u0, cases, streams)]
    for _ in range(30):
        for p in probs:
            p.advance(17, "swept")
    for p, s, u in zip(probs, specs, u0):
        assert np.array_equal(p.read(), _oracle(s, u, 30 * 17))
        p.close()


def test_capture_takes_the_replayable_route():
    """An advance captured by the caller and replayed three times: sequence
    numbers would repeat, so a captured advance runs the form without them."""
    torch = pytest.importorskip("torch")
    spec = spec_for("ks", "periodic", 1024)
    u0 = state_for(spec)
    stream = torch.cuda.Stream()
    with S.Problem(spec, u0, stream=stream) as p:
        p.advance(8, "swept")
        p.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            p.advance(20, "swept")
        with torch.cuda.stream(stream):
            for _ in range(3):
                g.replay()
        assert np.array_equal(p.read(), _oracle(spec, u0, 8 + 3 * 20))


def test_withheld_words_time_out_and_recover():
    spec = spec_for("heat", "periodic", 4099)
    u0 = state_for(spec)
    with S.Problem(spec, u0) as p:
        p.debug_withhold_flags(True, wait_limit_ns=100_000_000)
        t0 = time.perf_counter()
        p.advance(300, "swept")
        with pytest.raises(S.SweptError) as e:
            p.synchronize()
        assert e.value.status == S.ETIMEOUT
        assert time.perf_counter() - t0 < 30
        p.debug_withhold_flags(False)
        p.write(u0)
        p.advance(300, "swept")
        assert np.array_equal(p.read(), _oracle(spec, u0, 300))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_batch_of_whole_advances(dtype):
    """The batched resident launch: problems of one tile (their halos are their
    own points, over several periods for the smallest), of two, and of many,
    more tiles than the launch has blocks, advances of one level, of an odd
    number, of one exchange exactly and of many; twice, the second time replayed
    from a graph with the rows exchanged."""
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    kinds = [("heat", "periodic"), ("heat", "reflective"), ("ks", "periodic")]
    sizes = [16, 21, 100, 735, 745, 1489, 1857, 2049, 4099, 30011, 100003]
    steps = [1, 3, 8, 64, 97, 130]
    cases = [(eq, bc, N, steps[(i + j) % 6]) for i, N in enumerate(sizes) for j, (eq, bc) in enumerate(kinds)]
    cases += [("heat", "periodic", 3000 + 17 * i, 20 + i) for i in range(400)]
    specs = [spec_for(eq, bc, N) for eq, bc, N, _ in cases]
    u0 = [state_for(s, _np(dtype), seed=i) for i, s in enumerate(specs)]
    probs = [S.Problem(s, u, dtype, stream=stream) for s, u in zip(specs, u0)]
    with S.Batch(stream) as b:
        for _ in range(3):
            b.advance_ex(probs, [c[3] for c in cases], ["swept"] * len(cases), launch="graph")
        b.advance(probs, [c[3] for c in cases])
        b.synchronize()
        assert b.kernel_launches() == 4
    for (eq, bc, N, st), s, u, p in zip(cases, specs, u0, probs):
        assert np.array_equal(p.read(), _oracle(s, u, 4 * st)), (eq, bc, N, st)
        p.close()


@pytest.mark.parametrize("dtype,count,lo,hi", [
    ("f64", 1, 9001, 9002), ("f64", 5, 9000, 15000),            # short tiles
    ("f64", 60, 5000, 6000),                                    # the dataflow launch, default widths
    ("f64", 60, 15000, 16000), ("f64", 110, 15000, 16000), ("f64", 250, 15000, 16000),   # longer ones
    ("f32", 3, 3000, 9000), ("f32", 220, 15000, 16000)])
def test_batch_tile_lengths(dtype, count, lo, hi):
    """Batches on each side of the lines between tile lengths, with widths that
    the on-chip form does not use: every problem equals its classic advance."""
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    rng = np.random.default_rng(count)
    kinds = [("heat", "periodic"), ("ks", "periodic"), ("heat", "reflective")]
    specs = [spec_for(*kinds[i % 3], int(rng.integers(lo, hi))) for i in range(count)]
    steps = [int(rng.integers(17, 60)) for _ in specs]
    u0 = [state_for(s, _np(dtype), seed=i) for i, s in enumerate(specs)]
    probs = [S.Problem(s, u, dtype, stream=stream) for s, u in zip(specs, u0)]
    with S.Batch(stream) as b:
        b.advance_ex(probs, steps, ["swept"] * count, [S.fit_width(s.eq, s.n_points, 2048) for s in specs])
        b.synchronize()
    for s, u, st, p in zip(specs, u0, steps, probs):
        with S.Problem(s, u, dtype, stream=stream) as q:
            q.advance(st, "classic")
            assert np.array_equal(p.read(), q.read()), (s.eq, s.bc, s.n_points, st)
        p.close()

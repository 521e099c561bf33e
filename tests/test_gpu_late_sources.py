"""Source times far from 0: plans, the solve without allocation and solves that go
on after a bucket slot overflowed start at the first source's bucket like a plain solve.  From bucket 0
every tile would be clamped to the ring's last slot, in no order, which shows in
the number of visits; the bits are the oracle's either way."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_05694_gb300 as eik  # noqa: E402

DEV = "cuda:0"
SHAPES = [(300, 350), (48, 52, 60)]
T0 = 2e5


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2103_05694_gb300 import build
    build.build()
    eik.load_library()


def _problem(shape, t0):
    rng = np.random.Generator(np.random.PCG64(3))
    speed = rng.uniform(1.0, 4.0, shape)
    src = np.sort(rng.choice(speed.size, 12, replace=False)).astype(np.int64)
    return speed, src, t0 + rng.random(12)


def _bits(x):
    return np.ascontiguousarray(x).view(np.uint64)


def _plan(speed, src, times, opts):
    q = {"speed": torch.from_numpy(speed).to(DEV), "h": 0.5, "sources": torch.from_numpy(src).to(DEV),
         "src_t": torch.from_numpy(times).to(DEV)}
    plan = eik.Plan([q], opts)
    plan.enqueue()
    stats = plan.status()
    out = q["out"].cpu().numpy()
    plan.close()
    return out, stats


@pytest.mark.parametrize("shape", SHAPES)
def test_plan(shape):
    early = _plan(*_problem(shape, 0.0), {"counters": 1})[1]
    speed, src, times = _problem(shape, T0)
    want = oracle.fmm(speed, 0.5, src, times).t
    out, late = _plan(speed, src, times, {"counters": 1})
    assert np.array_equal(_bits(out), _bits(want))
    assert late["visits"] < 2 * early["visits"]
    assert np.array_equal(_bits(_plan(speed, src, times, None)[0]), _bits(want))


@pytest.mark.parametrize("shape", SHAPES)
def test_resumed_solve(shape):
    opts = {"counters": 1, "capacity": 16}
    visits = []
    for t0 in (0.0, T0):
        speed, src, times = _problem(shape, t0)
        r = eik.solve(torch.from_numpy(speed).to(DEV), 0.5, src, torch.from_numpy(times).to(DEV), opts=opts)
        assert r.stats["retries"] > 0
        visits.append(r.stats["visits"])
    assert np.array_equal(_bits(r.t.cpu().numpy()), _bits(oracle.fmm(speed, 0.5, src, times).t))
    assert visits[1] < 2 * visits[0]


@pytest.mark.parametrize("shape", SHAPES)
def test_noalloc(shape):
    visits = []
    for t0 in (0.0, T0):
        speed, src, times = _problem(shape, t0)
        dev = [torch.from_numpy(x).to(DEV) for x in (speed, src, times)]
        out = torch.full_like(dev[0], -1.0)
        stats = eik.eik_solve_noalloc(dev[0].data_ptr(), 0.5, speed.ndim, speed.shape, dev[1].data_ptr(),
                                      dev[2].data_ptr(), src.size, out.data_ptr(), {"counters": 1},
                                      torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        visits.append(stats["visits"])
    assert np.array_equal(_bits(out.cpu().numpy()), _bits(oracle.fmm(speed, 0.5, src, times).t))
    assert visits[1] < 2 * visits[0]


@pytest.mark.parametrize("opts", [None, {"arith": 1}, {"arith": 2}, {"counters": 1}, {"arith": 1, "window": 1}])
@pytest.mark.parametrize("shape", [(5, 6), (90, 110), (4, 4, 4), (20, 22, 25)])
def test_beyond_the_last_bucket(shape, opts):
    """Times of more than 2^30 bucket widths share the last bucket."""
    rng = np.random.Generator(np.random.PCG64(4))
    speed = rng.uniform(1.0, 4.0, shape)
    src = np.sort(rng.choice(speed.size, 9, replace=False)).astype(np.int64)
    times = 1e12 + rng.random(9)
    want = oracle.fmm(speed, 0.5, src, times).t
    r = eik.solve(torch.from_numpy(speed).to(DEV), 0.5, src, torch.from_numpy(times).to(DEV),
                  opts=dict(opts or {}, timeout_ms=5000))
    assert np.array_equal(_bits(r.t.cpu().numpy()), _bits(want))

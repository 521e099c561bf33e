"""Slab epochs that go on from the last epoch's fields, and solves whose first
source time lies far from 0 (the scheduler starts at its bucket): the oracle's
bits in every kernel and shape (no tolerance)."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_05694_gb300 as eik  # noqa: E402

DEV = "cuda:0"
OPTS = [{}, {"arith": 1}, {"arith": 2}, {"arith": 1, "tile": 2}, {"arith": 1, "k_delta": 0.5, "window": 1},
        {"capacity": 16, "arith": 1}]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2103_05694_gb300 import build
    build.build()
    eik.load_library()


def _channel(shape):
    """Slow cells with fast channels that wind through all slabs."""
    rng = np.random.Generator(np.random.PCG64(3))
    speed = 1.0 + rng.random(shape)
    speed[..., 1::6] *= 40.0
    speed[1::12] *= 40.0
    return speed


@pytest.mark.parametrize("opts", OPTS)
@pytest.mark.parametrize("shape,k", [((37, 50), 3), ((24, 9), 8), ((13, 11, 18), 3), ((9, 16, 9), 9)])
@pytest.mark.parametrize("t0", [0.0, 5e4])
def test_slabs(shape, k, t0, opts):
    speed = _channel(shape)
    src = np.array([2, speed.size - 3], dtype=np.int64)
    times = np.array([t0, t0 + 0.3])
    ref = oracle.fmm(speed, 0.7, src, times).t
    r = eik.solve_slabs(torch.from_numpy(speed).to(DEV), 0.7, src, k, src_t=times, opts=opts)
    torch.cuda.synchronize()
    assert np.array_equal(r.t.cpu().numpy().view(np.uint64), ref.view(np.uint64))
    assert r.stats["epochs"] >= 2


@pytest.mark.parametrize("opts", OPTS)
@pytest.mark.parametrize("shape", [(33, 70), (12, 17, 20)])
@pytest.mark.parametrize("spread", [0.0, 3.0, 1e4])
def test_late_sources(shape, spread, opts):
    p = synth.random_problem(9, shape, n_src=5, contrast=6.0, h=0.5)
    times = 2e4 + spread * np.random.Generator(np.random.PCG64(1)).random(5)
    ref = oracle.fmm(p.speed, p.h, p.sources, times).t
    r = eik.solve(torch.from_numpy(p.speed).to(DEV), p.h, p.sources, torch.from_numpy(times).to(DEV), opts=opts)
    torch.cuda.synchronize()
    assert np.array_equal(r.t.cpu().numpy().view(np.uint64), ref.view(np.uint64))

"""More tiles ready at once than a bucket slot has room for, in the kernels of
automatic options: a solve goes on with more room, a plan has the room that it had
with larger tiles.  A source in every tile (or in most) makes all of them ready in
bucket 0; slots have next_pow2(tiles / 4 + 4096) entries at first."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_05694_gb300 as eik  # noqa: E402

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2103_05694_gb300 import build
    build.build()
    eik.load_library()


def _lattice(shape, tile, part, seed):
    """A cell inside each of `part` of the tiles."""
    rng = np.random.Generator(np.random.PCG64(seed))
    at = np.meshgrid(*[np.arange(t // 2, n, t) for n, t in zip(shape, tile)], indexing="ij")
    cells = np.ravel_multi_index([a.ravel() for a in at], shape)
    return np.sort(cells[rng.random(cells.size) < part]).astype(np.int64)


def _bits(x):
    return np.ascontiguousarray(x).view(np.uint64)


def test_plan_keeps_its_room():
    """18,090 tiles of 8x8 (9,045 of 16x8, which fitted 16,384 entries)."""
    shape = (1080, 1072)
    src = _lattice(shape, (8, 8), 1.0, 1)
    speed = np.full(shape, 2.0)
    q = {"speed": torch.from_numpy(speed).to(DEV), "h": 1.0, "sources": torch.from_numpy(src).to(DEV)}
    plan = eik.Plan([q])
    plan.enqueue()
    plan.status()
    assert np.array_equal(_bits(q["out"].cpu().numpy()), _bits(oracle.fmm(speed, 1.0, src).t))
    plan.close()


def _one_bucket(shape):
    """A few slow rows raise the mean of h / v, and with it the bucket width, so far
    that the fast rest of the grid is one bucket."""
    speed = np.full(shape, 2.0)
    speed[-max(1, shape[0] // 20):] = 2e-3
    return speed


# part 1: the seeds overflow the slot; less: they fit, and the first visits' activations
# do not
@pytest.mark.parametrize("shape,tile,part", [((1024, 1024), (8, 8), 1.0), ((1024, 1024), (8, 8), 0.47),
                                             ((96, 96, 96), (4, 4, 4), 1.0), ((96, 96, 96), (4, 4, 4), 0.56)])
def test_front_kernel_goes_on(shape, tile, part):
    speed, src = _one_bucket(shape), _lattice(shape, tile, part, 2)
    r = eik.solve(torch.from_numpy(speed).to(DEV), 1.0, src)
    assert r.stats["retries"] > 0
    assert np.array_equal(_bits(r.t.cpu().numpy()), _bits(oracle.fmm(speed, 1.0, src).t))


@pytest.mark.parametrize("part", [1.0, 0.38])
def test_guided_kernel_goes_on(part):
    """41.8 million cells in 168,432 tiles of 8x8x4; the other kernel's bits."""
    shape = (347, 347, 347)
    speed = torch.from_numpy(_one_bucket(shape)).to(DEV)
    src = torch.from_numpy(_lattice(shape, (4, 8, 8), part, 3)).to(DEV)
    r = eik.solve(speed, 1.0, src)
    assert r.stats["retries"] > 0
    want = eik.solve(speed, 1.0, src, opts={"arith": 1}).t
    assert torch.equal(r.t.view(torch.int64), want.view(torch.int64))

"""The front kernel (8x8 and 4x4x4 tiles with live halos) and the guided kernel on
either side of the rule that chooses them: the oracle's bits at the edges of the
tiles, where fronts meet, with sources in halos and in batches of different
grids; the tile kernel's bits in volumes large enough for the guided kernel."""
import numpy as np
import pytest

import oracle
import synth

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


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


SHAPES = [(1, 1), (8, 8), (7, 9), (16, 8), (9, 17), (1, 33), (40, 3), (61, 75),
          (4, 4, 4), (3, 5, 4), (8, 4, 9), (1, 1, 9), (5, 1, 6), (14, 19, 23)]


@pytest.mark.parametrize("n_src", [1, 4, 12])
@pytest.mark.parametrize("shape", SHAPES)
def test_tile_edges_and_meeting_fronts(shape, n_src):
    n = int(np.prod(shape))
    p = synth.random_problem(11 + n_src, shape, n_src=min(n_src, n), contrast=20.0, h=0.4, src_t_max=0.6)
    ref = oracle.fmm(p.speed, p.h, p.sources, p.src_t).t
    for _ in range(3):                      # another schedule each time
        r = eik.solve(_dev(p.speed), p.h, _dev(p.sources), _dev(p.src_t))
        assert np.array_equal(r.t.cpu().numpy().view(np.uint64), ref.view(np.uint64))


@pytest.mark.parametrize("ndim", [2, 3])
def test_winding_channels(ndim):
    """A front that leaves and enters tiles again through every face."""
    shape = (50, 66) if ndim == 2 else (18, 22, 26)
    speed = np.full(shape, 1e-3)
    speed[..., ::4, :] = 1.0
    speed[..., 2::8, -1] = speed[..., 1::8, -1] = speed[..., 3::8, -1] = 1.0
    speed[..., 5::8, 0] = speed[..., 6::8, 0] = speed[..., 7::8, 0] = 1.0
    ref = oracle.fmm(speed, 0.1, [0]).t
    r = eik.solve(_dev(speed), 0.1, [0])
    assert np.array_equal(r.t.cpu().numpy().view(np.uint64), ref.view(np.uint64))


@pytest.mark.parametrize("ndim", [2, 3])
def test_batch_of_different_grids(ndim):
    probs, want = [], []
    for k in range(11):
        shape = tuple(int(x) for x in np.random.Generator(np.random.PCG64(k)).integers(1, 40 if ndim == 2 else 14, ndim))
        p = synth.random_problem(k, shape, n_src=1, contrast=5.0, h=0.7)
        want.append(oracle.fmm(p.speed, p.h, p.sources).t)
        probs.append({"speed": _dev(p.speed), "h": p.h, "sources": _dev(p.sources),
                      "out": torch.empty(shape, dtype=torch.float64, device=DEV)})
    eik.eik_solve_batched(probs)
    for q, w in zip(probs, want):
        assert np.array_equal(q["out"].cpu().numpy().view(np.uint64), w.view(np.uint64))


@pytest.mark.parametrize("n", [8, 9])
def test_large_batches_equal_the_tile_kernel(n):
    """39.1 and 44.0 million cells: the front kernel's and the guided kernel's side."""
    p = synth.random_problem(7, (167, 171, 171), n_src=1, contrast=6.0)
    speed = _dev(p.speed)
    rng = np.random.Generator(np.random.PCG64(n))
    srcs = [torch.tensor([int(rng.integers(p.speed.size))], device=DEV) for _ in range(n)]
    outs = [[torch.empty_like(speed) for _ in srcs] for _ in range(2)]
    for o, opts in zip(outs, (None, {"arith": 1})):
        eik.eik_solve_batched([{"speed": speed, "h": p.h, "sources": s, "out": t} for s, t in zip(srcs, o)], opts)
    for a, b in zip(*outs):
        assert torch.equal(a.view(torch.int64), b.view(torch.int64))


@pytest.mark.parametrize("n_grids", [1, 7, 12, 40])
def test_look_ahead_in_2d(n_grids):
    """Few grids: tiles start before a front reaches them.  Many: they don't (their
    fronts are in more tiles than there are CTAs), and more CTAs share the tiles.  Slow walls keep fronts away
    from tiles that wait for them."""
    speed = np.full((420, 600), 1.0)
    speed[::24, 5:] = speed[12::24, :-5] = 1e-4
    ref = oracle.fmm(speed, 0.5, [7]).t
    dev = _dev(speed)
    probs = [{"speed": dev, "h": 0.5, "sources": torch.tensor([7], device=DEV), "out": torch.empty_like(dev)}
             for _ in range(n_grids)]
    eik.eik_solve_batched(probs)
    for q in probs:
        assert np.array_equal(q["out"].cpu().numpy().view(np.uint64), ref.view(np.uint64))

"""The warp-per-tile adjoint at the edges of its tiles (16x16 in 2D, 8x4x4 in 3D),
with shared and own models, where its divisions leave the integer path, and when a
bucket slot overflows: the gradient equals the oracle's bit for bit (no tolerance:
both sides do the same roundings in the same order)."""
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


def _check(speeds, h, srcs, seed, slowness=False):
    rng = np.random.Generator(np.random.PCG64(seed))
    dev = {id(v): torch.from_numpy(1.0 / v if slowness else v).to(DEV) for v in speeds}
    probs, gs, grads, want = [], [], [], []
    for v, src in zip(speeds, srcs):
        used = 1.0 / (1.0 / v) if slowness else v
        t = oracle.fmm(used, h, src).t
        g = np.where(rng.random(v.shape) < 0.3, rng.standard_normal(v.shape), 0.0)
        want.append(oracle.adjoint(used, h, src, t, g)[1])
        probs.append({"speed": dev[id(v)], "h": h, "sources": torch.from_numpy(src).to(DEV),
                      "out": torch.from_numpy(t).to(DEV)})
        gs.append(torch.from_numpy(g).to(DEV))
        grads.append(torch.full(v.shape, np.nan, dtype=torch.float64, device=DEV))
    flags = eik.ADJ_TILES | (eik.SLOWNESS_INPUT if slowness else 0)
    st = eik.eik_adjoint(probs, gs, grads, opts={"sched_flags": flags, "timeout_ms": 10000})
    torch.cuda.synchronize()
    for got, w in zip(grads, want):
        assert np.array_equal(got.cpu().numpy().view(np.uint64), w.view(np.uint64))
    assert st["good"] == st["evals"] == sum(v.size for v in speeds)


@pytest.mark.parametrize("slowness", [False, True])
@pytest.mark.parametrize("shape", [(16, 16), (15, 17), (17, 15), (1, 33), (32, 16), (4, 4, 8), (5, 3, 9),
                                   (3, 5, 7), (8, 8, 16), (1, 1, 17), (9, 1, 1)])
def test_tile_edges(shape, slowness):
    a, b = (synth.random_problem(s, shape, n_src=1, contrast=8.0).speed for s in (1, 2))
    srcs = [np.array([k % a.size], dtype=np.int64) for k in (0, a.size - 1, a.size // 2)]
    _check([a, b, a], 0.75, srcs, 3, slowness)      # a is shared, b is not


@pytest.mark.parametrize("h", [1e-150, 1e150])
def test_extreme_scales(h):
    v = synth.random_problem(5, (19, 23), n_src=1, contrast=6.0).speed
    _check([v, v], h, [np.array([0], dtype=np.int64), np.array([200], dtype=np.int64)], 7)


def test_slot_overflow_goes_on():
    """3000 tiles that are all ready at once and share a bucket: more than a
    slot's first 2048 entries."""
    v = np.full((800, 960), 2.0)
    y, x = np.mgrid[0:800:16, 0:960:16]
    src = np.sort((y * 960 + x).ravel()).astype(np.int64)
    _check([v], 1.0, [src], 11)

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
    """One cell of `part` of the tiles, anywhere in it."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nt = [-(-n // t) for n, t in zip(shape, tile)]
    cells = []
    for k in np.ndindex(*nt):
        if rng.random() < part:
            at = [min(int(i * t + rng.integers(t)), n - 1) for i, t, n in zip(k, tile, shape)]
            cells.append(int(np.ravel_multi_index(at, shape)))
    return np.unique(np.array(cells, dtype=np.int64))


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

"""The adjoint of batches of unlike grids: the set-up runs over all cells in one loop
when the largest problem is far above the average one, else with a grid row per
problem.  The oracle's bits on both sides of that rule (no tolerance), and a large
grid is set up as fast beside many small ones as alone."""
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


@pytest.mark.parametrize("ndim", [2, 3])
@pytest.mark.parametrize("large_at", [0, 7, 60, None])
def test_uneven_batch_equals_oracle(ndim, large_at):
    rng = np.random.Generator(np.random.PCG64(17))
    top = 40 if ndim == 2 else 12
    shapes = [tuple(int(x) for x in rng.integers(1, top, ndim)) for _ in range(60)]
    if large_at is None:                      # twice the average at most
        shapes = [s for s in shapes if int(np.prod(s)) * 60 <= 2 * sum(int(np.prod(x)) for x in shapes)]
    else:                                     # more cells than threads
        shapes.insert(large_at, (613, 701) if ndim == 2 else (61, 83, 79))
    probs, gs, grads, want = [], [], [], []
    for k, shape in enumerate(shapes):
        p = synth.random_problem(k, shape, n_src=1, contrast=5.0, h=0.5)
        t = oracle.fmm(p.speed, p.h, p.sources).t
        g = rng.standard_normal(shape)
        want.append(oracle.adjoint(p.speed, p.h, p.sources, t, g)[1])
        probs.append({"speed": torch.from_numpy(p.speed).to(DEV), "h": p.h,
                      "sources": torch.from_numpy(p.sources).to(DEV), "out": torch.from_numpy(t).to(DEV)})
        gs.append(torch.from_numpy(g).to(DEV))
        grads.append(torch.full(shape, np.nan, dtype=torch.float64, device=DEV))
    st = eik.eik_adjoint(probs, gs, grads, opts={"sched_flags": eik.ADJ_TILES, "timeout_ms": 10000})
    torch.cuda.synchronize()
    for k, (got, w) in enumerate(zip(grads, want)):
        assert np.array_equal(got.cpu().numpy().view(np.uint64), w.view(np.uint64)), shapes[k]
    assert st["good"] == st["evals"] == sum(int(np.prod(s)) for s in shapes)


def test_large_grid_beside_small_ones():
    """Two per cent more cells; more than three times as long when each problem gets the
    blocks of the average one."""
    def best(shapes):
        speeds = [torch.full(s, 2.0, dtype=torch.float64, device=DEV) for s in shapes]
        probs = [{"speed": v, "h": 1.0, "sources": torch.zeros(1, dtype=torch.int64, device=DEV),
                  "out": torch.empty_like(v)} for v in speeds]
        eik.eik_solve_batched(probs)
        gs, grads = [torch.ones_like(v) for v in speeds], [torch.empty_like(v) for v in speeds]
        return min(eik.eik_adjoint(probs, gs, grads, opts={"sched_flags": eik.ADJ_TILES})["solve_ms"] for _ in range(4))
    large = (3000, 3000)
    assert best([large] + [(20, 25)] * 300) < 2.0 * best([large])

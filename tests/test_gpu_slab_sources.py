"""Slab decomposition with sources that other fronts reach before their own time, in
and beside the boundary rows: a source keeps its time in both slabs (the oracle's
bits, no tolerance)."""
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


@pytest.mark.parametrize("opts", [None, {"arith": 1}])
@pytest.mark.parametrize("shape", [(12, 9), (23, 41), (6, 2, 4), (7, 2, 10), (23, 3, 14), (9, 8, 7)])
@pytest.mark.parametrize("seed", range(4))
def test_late_sources_in_slabs(shape, seed, opts):
    p = synth.random_problem(300 + seed, shape, n_src=max(2, int(np.prod(shape)) // 6), contrast=(3.0, 300.0)[seed % 2],
                             h=0.5, src_t_max=(0.5, 5.0, 50.0, 1.0)[seed])
    ref = oracle.fmm(p.speed, p.h, p.sources, p.src_t).t
    speed = torch.from_numpy(p.speed).to(DEV)
    for k in (2, 3, shape[0] // 2, shape[0]):
        r = eik.solve_slabs(speed, p.h, p.sources, k, src_t=p.src_t, opts=opts)
        torch.cuda.synchronize()
        assert np.array_equal(r.t.cpu().numpy().view(np.uint64), ref.view(np.uint64)), k

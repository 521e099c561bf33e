"""The kernels that automatic options run, where the other GPU tests ask for the
kernel of explicit options: the full-size single grids (front kernel), and small
grids of every kind in the guided kernel, which takes 3D batches of 8 sources and 40
million cells or more (here a constant volume fills the batch up)."""
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


def _bits(x):
    return np.ascontiguousarray(x).view(np.uint64)


def test_layered_section_equals_oracle():
    p = synth.layered_2d_2301x751()
    ref = oracle.fmm(p.speed, p.h, p.sources).t
    speed = _dev(p.speed)
    for _ in range(3):                      # another schedule each time
        assert np.array_equal(_bits(eik.solve(speed, p.h, p.sources).t.cpu().numpy()), _bits(ref))


@pytest.mark.parametrize("n_src", [1, 8])
def test_checkerboard_equals_the_kernel_compared_with_the_oracle(n_src):
    """One source: the volume that the parity tests compare with the oracle."""
    p = synth.checker_3d_256()
    src = np.concatenate([p.sources, np.arange(1, n_src) * 1999999]).astype(np.int64)
    speed = _dev(p.speed)
    want = eik.solve(speed, p.h, src, opts={"arith": 1}).t
    for _ in range(2):
        assert torch.equal(eik.solve(speed, p.h, src).t.view(torch.int64), want.view(torch.int64))


SHAPES = [(1, 1, 1), (1, 1, 40), (1, 40, 1), (40, 1, 1), (4, 8, 8), (5, 9, 9), (3, 7, 7), (8, 16, 16), (9, 17, 15),
          (1, 33, 8), (4, 1, 65), (13, 20, 1), (2, 30, 31), (17, 12, 26)]


@pytest.mark.parametrize("h,contrast,late", [(1.0, 1.0, 0.0), (0.5, 20.0, 0.6), (1e-30, 50.0, 0.0), (1e40, 4.0, 0.5)])
def test_guided_kernel_equals_oracle(h, contrast, late):
    """contrast 1: every value ties with others, in and across tiles."""
    fill = torch.full((347, 347, 347), 2.0, dtype=torch.float64, device=DEV)
    probs, want = [{"speed": fill, "h": h, "sources": _dev(np.array([20000000])), "out": torch.empty_like(fill)}], [None]
    for k, shape in enumerate(SHAPES * 3):
        n = int(np.prod(shape))
        p = synth.random_problem(40 + k, shape, n_src=min((1, 3, 9)[k % 3], n), contrast=contrast, h=h,
                                 src_t_max=late * h)
        want.append(oracle.fmm(p.speed, p.h, p.sources, p.src_t).t)
        probs.append({"speed": _dev(p.speed), "h": h, "sources": _dev(p.sources), "src_t": _dev(p.src_t),
                      "out": torch.empty(shape, dtype=torch.float64, device=DEV)})
    probs = probs[1:20] + probs[:1] + probs[20:]
    want = want[1:20] + want[:1] + want[20:]
    eik.eik_solve_batched(probs)
    for q, w in zip(probs, want):
        if w is not None:
            assert np.array_equal(_bits(q["out"].cpu().numpy()), _bits(w)), w.shape

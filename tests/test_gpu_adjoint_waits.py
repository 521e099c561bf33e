"""The adjoint's waits: a CTA without a tile gives up when nothing is processed
anywhere for timeout_ms, not when its own turn is long in coming."""
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


@pytest.mark.parametrize("shape", [(12, 40000), (4, 4, 20000)])
def test_a_call_longer_than_the_limit(shape):
    """A strip: its tiles depend on each other in a chain of 2500, one at a time
    (some 20 us each), while the other CTAs wait ten times as long as the limit."""
    speed = np.full(shape, 2.0)
    src = np.array([0], dtype=np.int64)
    t = oracle.fmm(speed, 0.5, src).t
    g = np.zeros(shape)
    g.reshape(-1)[-1] = 1.0
    want = oracle.adjoint(speed, 0.5, src, t, g)[1]
    grad = torch.full(shape, np.nan, dtype=torch.float64, device=DEV)
    probs = [{"speed": torch.from_numpy(speed).to(DEV), "h": 0.5, "sources": torch.from_numpy(src).to(DEV),
              "out": torch.from_numpy(t).to(DEV)}]
    st = eik.eik_adjoint(probs, [torch.from_numpy(g).to(DEV)], [grad],
                         opts={"sched_flags": eik.ADJ_TILES, "timeout_ms": 2})
    torch.cuda.synchronize()
    assert st["solve_ms"] > 10.0            # else the limit was not passed
    assert np.array_equal(grad.cpu().numpy().view(np.uint64), want.view(np.uint64))

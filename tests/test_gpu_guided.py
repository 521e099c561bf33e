"""The guided tile kernel (the default of lean solves) and the integer d-bar it
evaluates: d-bar against the oracle's bisection from next to a source to far
from it and across binades; solves at the edges of the kernel's tiles, at
extreme scales and with exact ties, against the oracle; the shapes of large
volumes against the tile kernel that explicit options select."""
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


def _bits_equal(got, ref, what=""):
    g, e = got.view(np.uint64), ref.view(np.uint64)
    assert np.array_equal(g, e), f"{what}: {int((g != e).sum())} differ"


def _minima(rng, n, ratio, r, d):
    """Axis minima about `ratio` update lengths r from zero: anywhere, just below
    and on a power of two, equal, at the ends of the active range, absent."""
    s0 = r * ratio * rng.uniform(0.7, 1.4, n)
    pow2 = 2.0 ** np.floor(np.log2(s0))
    s0 = np.where(rng.random(n) < 0.2, pow2 * (1.0 - 1e-3 * rng.random(n) ** 3), s0)
    s0 = np.where(rng.random(n) < 0.1, pow2, s0)
    out = [s0]
    for _ in range(d - 1):
        b = s0 + r * 1.5 * rng.random(n) ** 2
        k = rng.integers(0, 12, n)
        b = np.where(k == 0, s0, b)
        b = np.where(k == 1, np.inf, b)
        b = np.where(k == 2, s0 + r * (1.0 + 1e-9 * rng.uniform(-1, 1, n)), b)
        out.append(b)
    out = np.stack(out, 1)
    return np.take_along_axis(out, rng.random(out.shape).argsort(1), 1)


@pytest.mark.parametrize("ratio", [1.3, 3.0, 20.0, 500.0, 1e5, 1e8])
def test_dbar_2d_equals_bisection(ratio):
    rng = np.random.Generator(np.random.PCG64(int(ratio * 10)))
    n = 3000
    v = rng.uniform(1.0, 4.0, n)
    a = _minima(rng, n, ratio, 1.25 / v, 2)
    got = eik.eik_eval_update(0, _dev(v), 1.25, _dev(a[:, 0]), _dev(a[:, 1])).cpu().numpy()
    want = np.array([oracle.dbar_bisect(a[i], oracle.cell_c(v[i], 1.25)) for i in range(n)])
    _bits_equal(got, want, f"ratio {ratio}")


@pytest.mark.parametrize("ratio", [1.3, 20.0, 1e4])
def test_dbar_3d_equals_bisection(ratio):
    """Cell 0 of a 2x2x2 grid whose three neighbours are sources."""
    rng = np.random.Generator(np.random.PCG64(int(ratio * 10) + 1))
    n = 400
    v = rng.uniform(1.0, 4.0, n)
    a = _minima(rng, n, ratio, 1.25 / v, 3)
    probs = []
    for i in range(n):
        keep = np.isfinite(a[i])
        probs.append({"speed": torch.full((2, 2, 2), float(v[i]), dtype=torch.float64, device=DEV), "h": 1.25,
                      "sources": _dev(np.array([1, 2, 4])[keep]), "src_t": _dev(a[i][keep]),
                      "out": torch.empty((2, 2, 2), dtype=torch.float64, device=DEV)})
    eik.eik_solve_batched(probs)
    got = np.array([q["out"].view(-1)[0].item() for q in probs])
    want = np.array([oracle.dbar_bisect(a[i], oracle.cell_c(v[i], 1.25)) for i in range(n)])
    _bits_equal(got, want, f"ratio {ratio}")


SHAPES = [(1, 1), (7, 9), (8, 8), (9, 17), (1, 65), (64, 3), (50, 71),
          (4, 4, 4), (5, 3, 9), (1, 2, 33), (12, 13, 11)]


@pytest.mark.parametrize("n_src,h,contrast", [(1, 1.0, 1.0), (3, 1e-30, 50.0), (9, 1e40, 4.0)])
@pytest.mark.parametrize("shape", SHAPES)
def test_solves_equal_oracle(shape, n_src, h, contrast):
    p = synth.random_problem(70 + len(shape), shape, n_src=n_src, contrast=contrast, h=h,
                             src_t_max=0.5 * h if n_src > 1 else 0.0)
    ref = oracle.fmm(p.speed, p.h, p.sources, p.src_t).t
    for opts in (None, {"arith": 3, "k_delta": 2.0, "capacity": 16}):
        r = eik.solve(_dev(p.speed), p.h, _dev(p.sources), _dev(p.src_t), opts=opts)
        _bits_equal(r.t.cpu().numpy(), ref, f"{shape} {opts}")


@pytest.mark.parametrize("n_src", [1, 9])
def test_large_volumes_equal_the_tile_kernel(n_src):
    """2^23 cells or more take 8x4x4 tiles (one front) or 8x8x4 (many)."""
    p = synth.random_problem(80 + n_src, (203, 205, 206), n_src=n_src, contrast=6.0)
    speed, src = _dev(p.speed), _dev(p.sources)
    a = eik.solve(speed, p.h, src).t
    b = eik.solve(speed, p.h, src, opts={"arith": 1}).t
    assert torch.equal(a.view(torch.int64), b.view(torch.int64))

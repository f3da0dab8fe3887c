"""GPU: every transform variant at the lengths where it can go wrong, against the oracle.

* The run-time plans: one length per radix (2 .. 16) and products of two and three of them, along each axis.
* The x1 turn's register variant (n1 = 64 .. 512 with enough lines): line counts that leave its last block
  part-filled, tau alone and tau with sigma (operator G), both schemes.
* The FP32 register passes along x2 and x3 (64: direct loads, 128 .. 512: tensor-map tiles): half spectra that
  leave the last tile part-filled, the real-direction operators and G^W.

FP64 fields within 1e-9 (the parity bar of test_gpu_parity).  FP32 fields against the oracle: two iterations are
four transforms each of at most log2(N) <= 20 butterfly levels, every level adding about one FP32 rounding
(6e-8) relative to the field's largest value, and the phases' law once: 2 x 4 x 20 x 6e-8 < 1e-5; the bar is 2e-5.
"""
import numpy as np
import pytest

from oracle import fftls_oracle as O
from paper_1412_8398_gb300 import microstructure as MS

pytestmark = pytest.mark.gpu
GREENS = {"MS": O.MS, "C": O.CENTERED, "W": O.WILLOT, "R": O.ROTATED}


@pytest.fixture(scope="module")
def solver():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_8398_gb300 import build, fftls
    build.build()
    s = fftls.Solver(0)
    yield s
    s.close()


def _check(solver, shape, green, scheme, precision):
    d = len(shape)
    ph = (np.random.default_rng(sum(shape)).random(shape) < 0.35).astype(np.uint8)
    lam, mu = MS.binary_moduli(8.0, d)
    eb = np.eye(d) * 0.4
    eb[0, 1] = eb[1, 0] = 0.3
    ref = O.solve(ph, lam, mu, eb, GREENS[green], O.ACCELERATED if scheme == "AS" else O.DIRECT, tol=0.0, max_iter=2)
    got = solver.solve(ph, lam, mu, eb, green, scheme, tol=0.0, max_iter=2, precision=precision, autotune=False)
    comps = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)] if d == 3 else [(0, 0), (1, 1), (0, 1)]
    want = np.stack([ref["strain"][i, j] for i, j in comps])
    bar = 1e-9 if precision == "fp64" else 2e-5 * np.abs(want).max()
    assert np.abs(got.strain - want).max() < bar
    np.testing.assert_allclose(got.eta_history, ref["eta_history"], rtol=1e-9 if precision == "fp64" else 1e-4)


@pytest.mark.parametrize("axis", range(3))
@pytest.mark.parametrize("n", [2, 5, 6, 9, 10, 12, 15, 16, 24, 25, 27, 32, 48, 75, 80, 90, 96, 100, 135, 144, 160, 250,
                               1024, 1080])
def test_run_time_plans(solver, axis, n):
    shape = [3, 4, 5]
    shape[axis] = n
    _check(solver, tuple(shape), "R", "AS", "fp64")
    _check(solver, tuple(shape), "W", "DS", "fp32")


@pytest.mark.parametrize("n1,n2,n3", [(64, 27, 50), (128, 25, 27), (256, 15, 25), (512, 9, 25)])
@pytest.mark.parametrize("green,scheme", [("R", "AS"), ("C", "DS"), ("MS", "AS"), ("MS", "DS")])
def test_turn_lines(solver, n1, n2, n3, green, scheme):
    for precision in ("fp64", "fp32"):
        _check(solver, (n3, n2, n1), green, scheme, precision)


@pytest.mark.parametrize("n", [64, 128, 256, 512])
@pytest.mark.parametrize("green", ["C", "R", "W"])
def test_register_passes(solver, n, green):
    for shape in ((n, 3, 18), (3, n, 18), (n, n if n < 256 else 64, 5)):
        _check(solver, shape, green, "AS", "fp32")


@pytest.mark.parametrize("shape", [(64, 128, 18), (128, 64, 10), (20, 64, 64)])
@pytest.mark.parametrize("green", ["R", "W", "MS"])
def test_grouped_register_kernels(solver, shape, green):
    """Grouped samples (the sample is a dimension of the tensor maps, and of the turn's grid) give bit for bit what
    each gives alone."""
    rng = np.random.default_rng(7)
    batch = []
    for i in range(3):
        lam, mu = MS.binary_moduli(4.0 + 5 * i, 3)
        batch.append({"phase": (rng.random(shape) < 0.3).astype(np.uint8), "lam": lam, "mu": mu,
                      "eps_bar": np.diag([1.0, 0.2 * i, -0.1]), "green": green, "scheme": "AS"})
    kw = dict(tol=1e-6, max_iter=60, precision="fp32_refine64", autotune=False)
    res, _ = solver.solve_batched(batch, concurrency=1, want_strain=True, **kw)
    for b, r in zip(batch, res):
        q = solver.solve(b["phase"], b["lam"], b["mu"], b["eps_bar"], green, "AS", raise_on_error=False, **kw)
        assert (r.status, r.iterations) == (q.status, q.iterations)
        assert np.array_equal(r.strain, q.strain)

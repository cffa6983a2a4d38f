"""The smoothing-length solve from bad first guesses and over its store's limits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2302_12727_gb300 import Transport, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def _clumps(n, rng):
    """A third of the particles each in a background, in clumps and in points of clumps: h
    varies by two hundred, and the cells of the mean density hold hundreds of particles."""
    a = rng.uniform(0, 1, (3, n - 2 * (n // 3)))
    c = rng.uniform(0.2, 0.8, (3, 4))
    b = c[:, rng.integers(0, 4, n // 3)] + 0.02 * rng.normal(size=(3, n // 3))
    d = c[:, rng.integers(0, 4, n // 3)] + 0.002 * rng.normal(size=(3, n // 3))
    return np.mod(np.concatenate([a, b, d], axis=1), 1.0)


def _bound(o, x, precision):
    """How far the root may be, relative to h.  The float phase ends where |f| <= 1e-6 h or the
    Newton step is below 2e-6 h, f = h - eta omega^(-1/3), and its sums round at 4e-7, all over
    f' = sum q |w'(q)| / (3 sum w(q)), which is small at the edge of a clump; the double one is exact to rounding."""
    if precision == "fp64":
        return 1e-12
    off, cols = o.pairs()
    i = np.repeat(np.arange(len(o.h)), np.diff(off))
    d = x[:, cols] - x[:, i]
    d -= np.round(d)
    q = np.sqrt((d * d).sum(0)) / (oracle.H_OVER_h * o.h[i])
    u, v = np.maximum(1 - q, 0), np.maximum(0.5 - q, 0)
    S = 0.5 + np.bincount(i, u ** 3 - 4 * v ** 3, len(o.h))
    fp = np.bincount(i, q * (3 * u ** 2 - 12 * v ** 2), len(o.h)) / (3 * S)
    return np.maximum(1e-6 / fp, 2e-6) + 4e-7 / fp


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [3001, 30000])
def test_h_from_the_guesses_of_other_places(n, precision):
    """Rebuilds whose particles have changed places: every first guess is the h of somewhere
    else, far too large or far too small."""
    _need_gpu()
    rng = np.random.default_rng(n)
    x = _clumps(n, rng)
    o = oracle.Oracle(x, np.full(n, 1.0 / n), None, n_groups=1)
    off, cols = o.pairs()
    count = np.diff(off)
    tol = _bound(o, x, precision)
    t = Transport(x, None, None, n_groups=1, precision=precision)
    for _ in range(3):
        assert (np.abs(t.h.cpu().numpy() / o.h - 1) <= tol).all()
        goff, gcols = t.pairs()
        assert np.array_equal(np.diff(goff.cpu().numpy()), count)
        key = np.repeat(np.arange(n), count) * n + cols
        gkey = np.repeat(np.arange(n), count) * n + gcols.cpu().numpy()
        assert np.array_equal(np.sort(gkey), np.sort(key))
        perm = rng.permutation(n)
        t.rebuild(x[:, perm])
        t.rebuild(x)
    t.close()


def test_h_of_a_support_that_overflows_the_store():
    """Particles in tight knots of 150: the support of a knot's neighbours holds more than the
    store, whatever the guess."""
    _need_gpu()
    rng = np.random.default_rng(11)
    g = W.jittered_lattice(10, 0.2, rng)
    knots = np.concatenate([g[:, k:k + 1] + 1e-3 * rng.normal(size=(3, 150)) for k in (111, 555)], axis=1)
    x = np.concatenate([g, knots], axis=1)
    n = x.shape[1]
    o = oracle.Oracle(x, np.full(n, 1.0 / n), None, n_groups=1)
    for precision in ("fp32", "fp64"):
        tol = _bound(o, x, precision)
        t = Transport(x, None, None, n_groups=1, precision=precision)
        assert (np.abs(t.h.cpu().numpy() / o.h - 1) <= tol).all()
        t.rebuild(x)
        assert (np.abs(t.h.cpu().numpy() / o.h - 1) <= tol).all()
        t.close()

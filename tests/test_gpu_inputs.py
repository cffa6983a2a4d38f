"""Inputs at and beyond the edge of what the calls accept."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2302_12727_gb300 import RTError, Transport, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("periodic", [True, False])
def test_positions_out_of_the_box_are_refused(precision, periodic):
    """One particle (or all of them) several boxes away, just outside, infinite or NaN on either
    axis: RT_ERR_INVALID from both searches, and the context then serves the valid set as before."""
    _need_gpu()
    rng = np.random.default_rng(2)
    x = W.jittered_lattice(12, 0.2, rng)
    t = Transport(x, None, None, n_groups=1, precision=precision, periodic=periodic)
    h = t.h.clone()
    for axis in range(3):
        for v in (1.0, -1e-3, 2.5, -1.5, 1e9, -1e300, np.inf, -np.inf, np.nan):
            bad = x.copy()
            bad[axis, 700 + axis] = v
            with pytest.raises(RTError, match="RT_ERR_INVALID"):
                t.rebuild(bad)
            with pytest.raises(RTError, match="RT_ERR_INVALID"):
                t.rebuild_given_h(h, x=bad)
    with pytest.raises(RTError, match="RT_ERR_INVALID"):
        t.rebuild(np.full_like(x, 7.0))
    t.rebuild(x)
    assert torch.equal(t.h, h)
    t.close()


def _sources_set(rng, n=20000):
    """A background with clumps, and sources in both: those in clumps overflow their candidate list."""
    c = rng.uniform(0.2, 0.8, (3, 3))
    x = np.mod(np.concatenate([rng.uniform(0, 1, (3, n // 2)),
                               c[:, rng.integers(0, 3, n - n // 2)] + 0.01 * rng.normal(size=(3, n - n // 2))], axis=1), 1)
    xsrc = np.concatenate([c, rng.uniform(0, 1, (3, 5)), [[0.0, 0.999], [0.002, 0.5], [0.998, 0.001]]], axis=1)
    return x, np.round(xsrc * 2 ** 20) / 2 ** 20      # box lengths are added to it exactly


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_sources_outside_a_periodic_box_are_their_images(precision):
    """The same sources whole boxes away: the same smoothing lengths, norms and injection, bit by bit."""
    _need_gpu()
    rng = np.random.default_rng(8)
    x, xsrc = _sources_set(rng)
    S = xsrc.shape[1]
    L = rng.uniform(0.5, 2.0, (S, 1))
    shifts = [np.zeros((3, S))] + [rng.integers(-4, 5, (3, S)).astype(float) for _ in range(2)]
    shifts.append(np.where(np.arange(3)[:, None] == np.arange(S) % 3, -1.0, 0.0))
    out = []
    for d in shifts:
        t = Transport(x, None, xsrc + d, n_groups=1, precision=precision)
        U = t.state(np.zeros((1, 4, x.shape[1])))
        t.inject(U, 1.0, t.luminosities(L))
        out.append([t.source_h(), *t.source_norms(), U])
        t.close()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert torch.equal(a, b)


def test_sources_outside_an_open_box():
    """Sources beside a box without periodic images, near and far: the oracle's h_s, omega_s and injection."""
    _need_gpu()
    rng = np.random.default_rng(9)
    x, _ = _sources_set(rng, 6000)
    n = x.shape[1]
    xsrc = np.array([[1.02, 0.5, -0.1, 1.3, -2.0], [0.5, -0.03, 1.2, 1.1, 4.0], [0.5, 1.01, 0.5, -0.2, 3.0]])
    o = oracle.Oracle(x, np.full(n, 1.0 / n), xsrc, n_groups=1, periodic=False)
    s = o.sources()
    t = Transport(x, None, xsrc, n_groups=1, precision="fp64", periodic=False)
    # the tolerances of sources inside (exact roots, sums of up to thousands of weights)
    assert np.abs(t.source_h().cpu().numpy() / s.hs - 1).max() <= 1e-12
    assert np.abs(t.source_norms()[0].cpu().numpy() / s.omegas - 1).max() <= 1e-11
    U = t.state(np.zeros((1, 4, n)))
    t.inject(U, 1.0, t.luminosities(np.ones((xsrc.shape[1], 1))))
    ref = o.inject(np.zeros((1, 4, n)), 1.0, np.ones((xsrc.shape[1], 1)))
    ref = np.asarray(ref[0] if isinstance(ref, tuple) else ref)
    assert np.abs(U.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
    t.close()


@pytest.mark.parametrize("periodic", [True, False])
def test_source_positions_that_are_not_finite_are_refused(periodic):
    _need_gpu()
    rng = np.random.default_rng(10)
    x = W.jittered_lattice(12, 0.2, rng)
    for v in (np.nan, np.inf, -np.inf):
        for axis in range(3):
            xsrc = np.full((3, 2), 0.4)
            xsrc[axis, 1] = v
            with pytest.raises(RTError, match="RT_ERR_INVALID"):
                Transport(x, None, xsrc, n_groups=1, precision="fp64", periodic=periodic)


def _beamed(G, n, rng):
    """States from isotropic to beyond the closure's clip, |F| up to 1.2 c E (c = 1), E in [1/2, 1]."""
    U = np.zeros((G, 4, n))
    U[:, 0] = rng.uniform(0.5, 1.0, (G, n))
    d = W.random_unit_vectors(G * n, rng).reshape(3, G, n).transpose(1, 0, 2)
    U[:, 1:] = rng.uniform(0, 1.2, (G, 1, n)) * U[:, :1] * d
    return U.astype(np.float32).astype(np.float64)


# the squares of 2^63 reach the top of the float range; the HLL wave speeds square F x A, and so reach
# neither as far down (F A of 2^-63) nor beyond |F| = 2^64
@pytest.mark.parametrize("riemann,powers", [("glf", (-50, 62, 63, 64, 100)), ("hll", (62, 63))])
@pytest.mark.parametrize("variant", [(0, 0, 0), (1, 1, 1), (2, 1, 2)])
@pytest.mark.parametrize("side,G", [(8, 2), (24, 3)])
def test_float_step_scales_over_the_exponent_range(side, G, variant, riemann, powers):
    """The step is homogeneous of degree one, and a power of two is exact: a scaled state gives the scaled
    result to a few roundings, in the plain step and with time bins."""
    _need_gpu()
    rng = np.random.default_rng(side)
    x = W.jittered_lattice(side, 0.2, rng)
    n = x.shape[1]
    U0 = _beamed(G, n, rng)
    t = Transport(x, None, None, n_groups=G, precision="fp32", riemann=riemann)
    t.set_tuning(*variant)
    dt = 0.2 * t.diagnostics()["dx_min"]
    t.set_time_bins(rng.integers(0, 3, n).astype(np.int32), dt_min=dt)
    base = None
    for k in (0,) + powers:
        a, b = t.state(np.ldexp(U0, k)), t.state(np.ldexp(U0, k))
        t.step(a, dt)
        t.step_bins(b)
        out = [np.ldexp(v.cpu().numpy().astype(np.float64), -k) for v in (a, b)]
        base = base or out
        for v, w in zip(out, base):
            assert np.abs(v - w).max() <= 1e-6 * np.abs(w).max(), k
    t.close()


@pytest.mark.parametrize("power", [505, 512, 700])
def test_double_step_scales_beyond_the_squares_of_the_states(power):
    _need_gpu()
    rng = np.random.default_rng(7)
    x = W.jittered_lattice(8, 0.2, rng)
    U0 = _beamed(2, x.shape[1], rng)
    t = Transport(x, None, None, n_groups=2, precision="fp64")
    a, b = t.state(U0), t.state(np.ldexp(U0, power))
    t.step(a, 0.01)
    t.step(b, 0.01)
    a, b = a.cpu().numpy(), np.ldexp(b.cpu().numpy(), -power)
    assert np.abs(a - b).max() <= 1e-14 * np.abs(a).max()
    t.close()


@pytest.mark.parametrize("precision,near,far,tol", [("fp64", -300, -560, 1e-12), ("fp32", -40, -70, 1e-5)])
def test_adjoint_of_states_with_little_energy(precision, near, far, tol):
    """|F| >> c E: the clipped closure is linear in E along F, so the gradient is the same for E of 2^near
    and of 2^far, up to terms of E / |F| (below the tolerance, a few roundings of sums of ~50 terms)."""
    _need_gpu()
    rng = np.random.default_rng(4)
    x = W.jittered_lattice(8, 0.2, rng)
    n = x.shape[1]
    U0 = _beamed(2, n, rng)
    U0[:, 1:] = W.random_unit_vectors(2 * n, rng).reshape(3, 2, n).transpose(1, 0, 2)
    lam = rng.normal(size=U0.shape)
    t = Transport(x, None, None, n_groups=2, precision=precision)
    out = []
    for k in (near, far):
        U = U0.copy()
        U[:, 0] = np.ldexp(U[:, 0], k)
        dU0, _ = t.adjoint(t.state(U), 1, 0.01, t.state(lam), None, None, 1)
        out.append(dU0.double().cpu().numpy())
    t.close()
    assert np.isfinite(out[1]).all()
    assert np.abs(out[0] - out[1]).max() <= tol * np.abs(out[0]).max()


def test_adjoint_slots_make_room_for_more_checkpoints():
    """A second adjoint with more checkpoints, on a device with little memory left: the context's optional
    buffers (the slots and pair geometry, about 500 MB here) go, and the result stays, to rounding."""
    _need_gpu()
    rng = np.random.default_rng(6)
    x = W.jittered_lattice(40, 0.2, rng)
    n = x.shape[1]
    U0, lam = _beamed(2, n, rng), rng.normal(size=(2, 4, n))
    n_sub = 160                                   # checkpoints of 4.1 MB each: 656 MB
    t = Transport(x, None, None, n_groups=2, precision="fp64")
    U, w = t.state(U0), t.state(lam)
    t.adjoint(U, 2, 1e-4, w, None, None, 1)
    sub = t.state(U0)
    t.subcycle(sub, 4, 1e-3)
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(max(free - (250 << 20), 1), dtype=torch.uint8, device="cuda")
    try:
        lean = t.adjoint(U, n_sub, 1e-4, w, None, None, 1)[0].cpu().numpy()
        again = t.state(U0)
        t.subcycle(again, 4, 1e-3)                # the captured graph held the geometry's address
        again = again.cpu().numpy()
    finally:
        del hold
        torch.cuda.empty_cache()
    t.rebuild(x)
    full = t.adjoint(U, n_sub, 1e-4, w, None, None, 1)[0].cpu().numpy()
    t.close()
    # the two evaluation orders differ by a few roundings a step
    assert np.abs(lean - full).max() <= n_sub * 1e-14 * np.abs(full).max()
    assert np.abs(again - sub.cpu().numpy()).max() <= 1e-13 * np.abs(again).max()


@pytest.mark.parametrize("G,threads", [(1, 1), (3, 3), (4, 4), (5, 3), (7, 4), (9, 3)])
def test_threads_per_particle_are_those_of_the_launch(G, threads):
    """Groups run in even chunks of at most four: 5 as 3 + 2, 7 as 4 + 3, 9 as 3 + 3 + 3."""
    _need_gpu()
    x = W.jittered_lattice(8, 0.2, np.random.default_rng(1))
    t = Transport(x, None, None, n_groups=G, precision="fp32")
    assert t.diagnostics()["threads_per_particle"] == threads
    t.close()

"""Dispatch branches of the float kernels and of the source search: every path of a rule against
the general one, bit by bit where only the launch differs, else against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2302_12727_gb300 import Transport, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def _state(G, n, rng):
    U = np.zeros((G, 4, n))
    U[:, 0] = rng.uniform(0.1, 1.0, size=(G, n))
    U[:, 1:] = 0.6 * U[:, :1] * rng.uniform(-1, 1, size=(G, 3, n))
    return U


# side 12: the wide gradient and gather (fewer than eight warps per SM); side 24: the kernels of
# larger sets for three groups and more, and, with HLL, the block that keeps the table in shared
# memory (two batches of 32 pairs for each of its warps); 7 and 9 groups are 4 + 3 and 3 + 3 + 3
@pytest.mark.parametrize("side,G,riemann", [(12, 1, "glf"), (12, 3, "glf"), (12, 4, "glf"), (24, 1, "hll"),
                                            (24, 2, "hll"), (24, 4, "hll"), (24, 7, "glf"), (9, 9, "hll")])
def test_default_kernels_equal_the_direct_ones(side, G, riemann):
    """Direct loads, one thread per particle, against the default variants: same bits."""
    _need_gpu()
    rng = np.random.default_rng(100 * side + G)
    x = W.poisson_sine_density(side ** 3, rng)
    xsrc = rng.uniform(0, 1, (3, 2))
    t = Transport(x, None, xsrc, n_groups=G, precision="fp32", riemann=riemann)
    dt = 0.3 * t.diagnostics()["dx_min"]
    U0 = _state(G, side ** 3, rng)
    L = t.luminosities(rng.uniform(0.5, 2.0, (2, G)))
    out = []
    for variant in ((0, 0, 0), (2, 1, 2)):
        t.set_tuning(*variant)
        U = t.state(U0)
        t.subcycle(U, 3, dt, L, None)
        V = t.state(U0)
        for _ in range(3):
            t.step(V, dt, L, None)
        assert torch.equal(U, V)
        out.append(U)
    assert torch.equal(out[0], out[1])
    assert t.diagnostics()["wait_timeouts"] == 0
    t.close()


def test_sources_with_and_without_a_candidate_list():
    """Sources in clumps, where the candidates of the first guess overflow the list, beside
    sources in the field, cold and warm: h_s, omega_s and the octant sums of the oracle."""
    _need_gpu()
    rng = np.random.default_rng(5)
    n = 20000
    c = rng.uniform(0.2, 0.8, (3, 3))
    x = np.mod(np.concatenate([rng.uniform(0, 1, (3, n // 2)),
                               c[:, rng.integers(0, 3, n - n // 2)] + 0.01 * rng.normal(size=(3, n - n // 2))], axis=1), 1)
    xsrc = np.concatenate([c, np.mod(c + 0.012, 1), rng.uniform(0, 1, (3, 3))], axis=1)
    o = oracle.Oracle(x, np.full(n, 1.0 / n), xsrc, n_groups=1)
    s = o.sources()
    t = Transport(x, None, xsrc, n_groups=1, precision="fp64")
    for _ in range(2):
        # the root is exact to rounding (1e-15); sums of up to ~100 weights round at 1e-14
        assert np.abs(t.source_h().cpu().numpy() / s.hs - 1).max() <= 1e-12
        om, _ = t.source_norms()
        assert np.abs(om.cpu().numpy() / s.omegas - 1).max() <= 1e-12
        t.rebuild(x)
    U = t.state(np.zeros((1, 4, n)))
    t.inject(U, 1.0, t.luminosities(np.ones((9, 1))))
    assert t.energy(U)[0] == pytest.approx(9.0, rel=1e-12)
    ref = o.inject(np.zeros((1, 4, n)), 1.0, np.ones((9, 1)))
    ref = np.asarray(ref[0] if isinstance(ref, tuple) else ref)
    assert np.abs(U.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
    t.close()

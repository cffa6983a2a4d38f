"""The double path's kernels that keep the pair geometry, against the oracle and each other.

Tolerances are those of the parity tests (the rounding bound of ~50-term neighbour sums);
the adjoint of two evaluation orders agrees to the rounding of the same sums, 1e-12 of the
largest value.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2302_12727_gb300 import Transport, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def _state(G, n, rng, c=1.0):
    U = np.zeros((G, 4, n))
    U[:, 0] = rng.uniform(0.5, 1.5, (G, n))
    U[:, 1:] = rng.uniform(0, 1.2, (G, 1, n)) * c * U[:, None, 0] * W.random_unit_vectors(G * n, rng).T.reshape(
        G, n, 3).transpose(0, 2, 1)
    return U


def _close(g, o):
    """Per element within 1e-12 |o| + 1e-14 of the group's largest value."""
    scale = np.abs(o).reshape(o.shape[0], -1).max(1).reshape(-1, *([1] * (o.ndim - 1)))
    return float((np.abs(g - o) / (1e-12 * np.abs(o) + 1e-14 * scale)).max())


# (side, G): four lanes a particle and group below 152 x 1024 of them, one lane above; 5 groups
# are two chunks (4 + 1)
@pytest.mark.parametrize("side,G", [(9, 1), (11, 5), (38, 3)])
def test_gradient_and_step_match_oracle(side, G):
    _need_gpu()
    rng = np.random.default_rng(side)
    x = W.jittered_lattice(side, 0.2, rng)
    n = x.shape[1]
    o = oracle.Oracle(x, np.full(n, 1.0 / n), None, n_groups=G)
    dt = 0.3 * ((o.V / (4 * np.pi / 3)) ** (1 / 3)).min()
    U0 = _state(G, n, rng)
    t = Transport(x, None, None, n_groups=G, precision="fp64")
    g = t.gradients(t.state(U0)).cpu().numpy()
    go = np.asarray(o.gradients(U0)).reshape(g.shape)
    assert _close(g, go) <= 10.0     # gradients divide the sums by h: one more digit of the scale
    U = t.state(U0)
    t.step(U, dt)
    assert _close(U.cpu().numpy(), o.run(U0, 1, dt)[0]) <= 1.0
    t.close()


@pytest.mark.parametrize("power", [-200, 200])
def test_step_scales_exactly_over_the_exponent_range(power):
    """The step is homogeneous of degree one: states of 1e-60 and 1e60 give the scaled result
    (the closure's ratio, reciprocal and root work on the squares of E and F)."""
    _need_gpu()
    rng = np.random.default_rng(7)
    x = W.jittered_lattice(8, 0.2, rng)
    U0 = _state(2, x.shape[1], rng)
    t = Transport(x, None, None, n_groups=2, precision="fp64")
    a, b = t.state(U0), t.state(np.ldexp(U0, power))
    t.step(a, 0.01)
    t.step(b, 0.01)
    assert _close(np.ldexp(b.cpu().numpy(), -power), a.cpu().numpy()) <= 1.0
    t.close()


@pytest.mark.parametrize("G", [2, 5])
def test_adjoint_without_slots_equals_adjoint_with_slots(G):
    """With little device memory left the adjoint evaluates each pair for both its particles
    and the transport computes the pair geometry in each kernel: same results to rounding."""
    _need_gpu()
    rng = np.random.default_rng(3)
    x = W.jittered_lattice(40, 0.2, rng)
    n = x.shape[1]
    xsrc = rng.uniform(0, 1, (3, 3))
    U0, lam = _state(G, n, rng), rng.normal(size=(G, 4, n))
    L = rng.uniform(0.5, 2, (3, G))

    def run():
        t = Transport(x, None, xsrc, n_groups=G, precision="fp64")
        out = [v.cpu().numpy() for v in t.adjoint(t.state(U0), 3, 1e-3, t.state(lam), t.luminosities(L), None, 2)]
        launches = t.diagnostics()["kernel_launches"]
        t.close()
        return out, launches

    full, n_full = run()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    # of what is left, the context's other buffers take 280 to 490 MB; the pair geometry (195 MB)
    # would need four times and the slots (295 to 590 MB) twice their size free
    hold = torch.empty(max(free - (700 << 20), 1), dtype=torch.uint8, device="cuda")
    try:
        lean, n_lean = run()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert n_lean < n_full           # two kernels a reverse step and chunk instead of five
    for a, b in zip(full, lean):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max()

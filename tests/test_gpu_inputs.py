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

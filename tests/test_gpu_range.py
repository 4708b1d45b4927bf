"""Sums of squares and moments far above FP32's range: a reconstruction scaled
by a power of two gives the scaled results, as sums in 64 bits do."""
import numpy as np
import pytest

from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu


def _plan(cp, N, Np, **kw):  # noqa: F811
    p = cp.Plan(cp.make_config(N, Np, **kw))
    p.load_intensities(np.ones((Np, N, N), np.float32), 0, np.arange(Np) * np.pi / Np)
    p.load_support(np.ones((N, N), np.uint8))
    return p


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 64])
@pytest.mark.parametrize("N", [16, 64, 96])
def test_twin_choice(cp, N, scale):  # noqa: F811
    """The second guess is the first one's twin, the third the first again:
    squared distances of 1e42 choose as those of 1e3 do.  Nothing lies in row
    and column 0, which x -> -x mod N leaves in place: the mass centre goes to
    N minus itself."""
    g = np.random.default_rng(N).random((2, N, N)).astype(np.float32) * np.float32(scale)
    g[:, 0] = g[:, :, 0] = 0.0
    twin = np.roll(g[:, ::-1, ::-1], (1, 1), (1, 2)).copy()
    plans = []
    for s in (g, twin, g):
        p = _plan(cp, N, 2)
        p.load_state(s, 1)  # one iteration on record, its error 0: kept in order
        plans.append(p)
    dst = _plan(cp, N, 2)
    assert cp.cpra_merge(plans, 3, 0, dst) == ([0, 1, 2], [False, True, False])
    for p in plans + [dst]:
        p.close()

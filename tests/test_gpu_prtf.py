"""The PRTF's ring sums do not depend on the order in which blocks and threads
add, and the PRTF of one guess is 1 in every ring."""
import numpy as np
import pytest

import synth
from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu


def _guesses(cp, N, Np, n):  # noqa: F811
    d = synth.make_case("tiny", N=N, Np=Np)
    out = []
    for i in range(n):
        p = cp.Plan(cp.make_config(N, Np, seed=i, hio_iters=2))
        p.load_intensities(d["I"], 0, d["thetas"])
        p.load_support(d["support"])
        p.iterate(3)
        out.append(p)
    dst = cp.Plan(cp.make_config(N, Np))
    dst.load_intensities(d["I"], 0, d["thetas"])
    return out, dst


@pytest.mark.parametrize("N,Np", [(96, 8), (128, 12)])
def test_the_same_merge_gives_the_same_prtf(cp, N, Np):  # noqa: F811
    g, dst = _guesses(cp, N, Np, 3)
    first = None
    for _ in range(6):
        prtf = np.empty((Np, N // 2), np.float32)
        cp.cpra_merge(g, 3, 0, dst, prtf)
        first = prtf if first is None else first
        assert np.array_equal(prtf, first)
    assert 0.05 < first.mean() < 1.0
    for p in g + [dst]:
        p.close()


@pytest.mark.parametrize("N", [16, 48, 64, 160, 700])
def test_one_guess_is_1_in_every_ring(cp, N):  # noqa: F811
    g, dst = _guesses(cp, N, 2, 1)
    prtf = np.empty((2, N // 2), np.float32)
    cp.cpra_merge(g, 1, 0, dst, prtf)
    assert np.abs(prtf - 1.0).max() < 2e-7  # |E| / |E|: an ulp of FP32 where the two square roots round apart
    for p in g + [dst]:
        p.close()

"""The one-launch Gauss-Seidel sweep at the sizes that run it."""
import numpy as np
import pytest

import oracle as O
import synth
from test_gpu_parity import TOL, _rel, cp  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,engine", [(16, 1), (32, 1), (48, 1), (96, 1), (160, 1), (320, 1),
                                      (64, 2), (128, 2), (256, 2)])
def test_one_angle_equals_the_jacobi_episode(cp, N, engine):  # noqa: F811
    """A carousel of one angle has no order, so a sweep of it is the Jacobi
    episode: the sweep kernels against the block-wide passes (1) and the fused
    engine (2), bit for bit, across the RAAR -> ER switch inside an episode."""
    d = synth.make_case("tiny", N=N, Np=1)
    out = []
    for sweep in (0, 1):
        p = cp.Plan(cp.make_config(N, 1, n_ei=3, seed=4, hio_iters=4, er_iters=2, engine=engine,
                                   update=cp.UPDATE_RAAR, wrap_mode=cp.WRAP_MIRROR, sweep=sweep))
        p.load_intensities(d["I"], 0, d["thetas"])
        p.load_support(d["support"])
        e = p.iterate(6, errors=True)
        out.append((p.result(cp.RESULT_STATE), e))
        p.close()
    assert np.array_equal(out[0][0], out[1][0])
    np.testing.assert_allclose(out[0][1], out[1][1], rtol=1e-5)  # FP32 partial sums of other threads


@pytest.mark.parametrize("N", [32, 64, 96, 128, 160, 256, 320])
@pytest.mark.parametrize("objt", [0, 1])
def test_sweep_against_the_oracle(cp, N, objt):  # noqa: F811
    """Two ER sweeps of five angles, five taps, MIRROR seam; a batch of an
    uneven pair of guesses (5 and 3 angles) ends where each ends alone."""
    d = synth.make_case("tiny", N=N, Np=5)
    kw = dict(n_ei=2, seed=3, hio_iters=0, er_iters=4, alpha=(0.1, 0.2, 0.4, 0.2, 0.1),
              wrap_mode=cp.WRAP_MIRROR, blend_target=objt, sweep=1)
    p = cp.Plan(cp.make_config(N, 5, **kw))
    p.load_intensities(d["I"], 0, d["thetas"])
    p.load_support(d["support"])
    e = p.iterate(4, errors=True)
    g = p.result(cp.RESULT_STATE)
    oc = O.OracleConfig(N=N, Np=5, n_ei=2, hio_iters=0, er_iters=4, seed=3, sweep=True,
                        alpha=kw["alpha"], wrap=kw["wrap_mode"], blend=objt)
    run = O.OracleRun.start(oc, d["I"], d["support"])
    for _ in range(2):
        run.sweep_episode()
    assert _rel(g, run.g).max() < TOL
    ref = np.array(run.errors)
    assert np.max(np.abs(e - ref) / ref) < TOL
    pair = []
    for Np in (5, 3):
        q = cp.Plan(cp.make_config(N, Np, **kw))
        q.load_intensities(d["I"][:Np], 0, d["thetas"][:Np])
        q.load_support(d["support"])
        pair.append(q)
    b = cp.Batch(pair)
    assert b.launches(4) == 2
    n0 = cp.cpra_launch_count()
    b.iterate(4)
    assert np.array_equal(pair[0].result(cp.RESULT_STATE), g)
    assert cp.cpra_launch_count() - n0 == 2 + 2  # the seeded starts, then the sweeps
    alone = cp.Plan(cp.make_config(N, 3, **kw))
    alone.load_intensities(d["I"][:3], 0, d["thetas"][:3])
    alone.load_support(d["support"])
    alone.iterate(4)
    assert np.array_equal(pair[1].result(cp.RESULT_STATE), alone.result(cp.RESULT_STATE))
    b.close()
    for q in pair + [alone, p]:
        q.close()

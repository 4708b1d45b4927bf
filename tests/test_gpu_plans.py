"""The line plans and kernel forms where no other test reaches them.

Refinement, merge and assembly at the sizes whose plans have idle lanes, blocks
of 10 or 24 columns, one line a warp or planes that do not fill a chunk,
against the 64-bit results of perf/cases.py; the fused engine's two-task form
(launches of more clusters than are resident with one task a warp) and sweeps
under a beamstop mask against the engines they must equal bit for bit.  The
bound of 2e-6 is three times the largest error of any size (6.6e-7, 360
angles)."""
import importlib.util
import os

import numpy as np
import pytest

import synth
from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BOUND = 2e-6


@pytest.fixture(scope="module")
def cases(cp):  # noqa: F811
    spec = importlib.util.spec_from_file_location("perf_cases", os.path.join(ROOT, "perf", "cases.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


def _rel(got, ref):
    ref = ref.to(got.device)
    return float((got.to(ref.dtype) - ref).norm() / ref.norm())


@pytest.mark.parametrize("N,Np,iters", [(16, 9, 3), (32, 12, 3), (48, 12, 3), (64, 12, 3), (96, 12, 3), (128, 12, 3), (160, 9, 2),
                                        (192, 9, 2), (256, 9, 2), (320, 7, 2), (384, 7, 2), (512, 5, 2), (640, 4, 2), (700, 4, 2), (768, 4, 1), (1024, 3, 1)])
def test_refinement(cases, N, Np, iters):
    case = dict(kind="refine", N=N, Np=Np, iters=iters)
    assert _rel(cases.run(cases.prepare(case, 1)), cases.exact(case, 1)) < BOUND


@pytest.mark.parametrize("N,Np", [(320, 7), (384, 7), (512, 7), (640, 5), (700, 5), (768, 4), (1024, 3)])
def test_assembly(cases, N, Np):
    case = dict(kind="assemble", N=N, Np=Np)
    assert _rel(cases.run(cases.prepare(case, 2)), cases.exact(case, 2)) < BOUND


@pytest.mark.parametrize("N", [32, 48, 96, 160, 192, 256, 320, 384, 512, 640, 700, 768])
def test_merge(cases, N):
    case = dict(kind="merge", N=N, Np=4, guesses=3, keep=3)
    got, ref = cases.run(cases.prepare(case, 1)), cases.exact(case, 1)
    assert _rel(got["spectra"], ref["spectra"]) < BOUND and _rel(got["volume"], ref["volume"]) < BOUND
    # a ring is a mean of ratios whose FP32 terms are right to 1e-6 of the
    # spectrum's magnitude there, to 1e-4 at its weakest pixels
    assert float((got["prtf"].double() - ref["prtf"]).abs().max()) < 1e-3
    twin = got["selected"] % 2
    assert np.array_equal(got["inverted"] != 0, twin != twin[0])


@pytest.mark.parametrize("N,Np", [(64, 700), (128, 400), (256, 200)])
@pytest.mark.parametrize("masked", [False, True])
def test_two_tasks_a_warp(cp, N, Np, masked):  # noqa: F811
    """The fused engine on more angles than fit with one task a warp equals the
    warp engine."""
    rng = np.random.default_rng(N)
    I = rng.random((Np, N, N)).astype(np.float32)
    S = rng.random((N, N)) < 0.4
    out = []
    for engine in (cp.ENGINE_FUSED, cp.ENGINE_WARP):
        p = cp.Plan(cp.make_config(N, Np, n_ei=2, seed=2, hio_iters=3, er_iters=2, update=cp.UPDATE_RAAR, engine=engine))
        if masked:
            p.load_mask(_stop(N))
        p.load_intensities(I, 0, np.arange(Np) * np.pi / Np)
        p.load_support(S.astype(np.uint8))
        e = p.iterate(5, errors=True)
        out.append((p.result(cp.RESULT_STATE), e))
        p.close()
    assert np.array_equal(out[0][0], out[1][0])
    np.testing.assert_allclose(out[0][1], out[1][1], rtol=1e-6)  # FP32 partial sums of other threads


def _stop(N):
    k = np.arange(N) - N // 2
    return (k[:, None] ** 2 + k[None, :] ** 2 > (N // 16) ** 2).astype(np.uint8)


@pytest.mark.parametrize("N,engine,members", [(32, 1, 1), (96, 1, 1), (96, 1, 24), (160, 1, 14), (64, 2, 1), (128, 2, 1), (256, 2, 1),
                                              (64, 2, 400), (128, 2, 160), (256, 2, 60)])
@pytest.mark.parametrize("masked", [False, True])
def test_sweeps_of_one_angle(cp, N, engine, members, masked):  # noqa: F811
    """A carousel of one angle has no order: sweeping it, alone or beside so
    many others that two tasks share a warp, is the Jacobi episode."""
    d = synth.make_case("tiny", N=N, Np=1)

    def plan(sweep):
        p = cp.Plan(cp.make_config(N, 1, n_ei=3, seed=4, hio_iters=4, er_iters=2, engine=engine, update=cp.UPDATE_RAAR, sweep=sweep))
        if masked:
            p.load_mask(_stop(N))
        p.load_intensities(d["I"], 0, d["thetas"])
        p.load_support(d["support"])
        return p

    ref = plan(0)
    ref.iterate(6)
    want = ref.result(cp.RESULT_STATE)
    group = [plan(1) for _ in range(members)]
    b = cp.Batch(group)
    b.iterate(6)
    for p in group[:3] + group[-3:]:
        assert np.array_equal(p.result(cp.RESULT_STATE), want)
    b.close()
    for p in group + [ref]:
        p.close()

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


@pytest.mark.parametrize("N,engine,sweep", [(32, 1, 0), (64, 3, 0), (64, 2, 0), (96, 0, 0), (160, 0, 0), (256, 2, 0), (512, 3, 0),
                                            (64, 2, 1), (96, 1, 1), (256, 2, 1)])
def test_iterates_and_errors(cp, N, engine, sweep):  # noqa: F811
    """Intensities up to 2^122: the sums of A^2 and of the error terms are far
    above FP32's largest number, single values are not (with nothing in the
    support HIO is g - beta g', whose spectrum stays below the amplitudes'
    order; positivity would add N / 10 of them up at the origin).  Scaling by a
    power of two commutes with every rounding."""
    rng = np.random.default_rng(N)
    I = rng.uniform(0.25, 1.0, (3, N, N)).astype(np.float32)
    g = (rng.random((3, N, N)) / N ** 2).astype(np.float32)
    out = []
    for k in (0, 61):
        p = cp.Plan(cp.make_config(N, 3, n_ei=2, hio_iters=4, engine=engine, sweep=sweep))
        p.load_intensities(I * np.float32(2.0 ** (2 * k)), 0, np.arange(3) * np.pi / 3)
        p.load_support(np.zeros((N, N), np.uint8))
        p.load_state(g * np.float32(2.0 ** k), 0)
        e = p.iterate(4, errors=True)
        out.append((p.result(cp.RESULT_STATE) / np.float32(2.0 ** k), e))
        p.close()
    assert np.array_equal(out[0][0], out[1][0])
    np.testing.assert_allclose(out[1][1], out[0][1], rtol=1e-10)  # sums in 64 bits or 48


@pytest.mark.parametrize("N,engine", [(32, 1), (64, 3), (64, 2), (96, 0), (256, 2), (512, 3)])
def test_mass_centres(cp, N, engine):  # noqa: F811
    """An object in the last eight rows: sum rho z is above FP32's largest
    number, sum rho and what the transforms hold are not (N times a row's sum
    is the largest)."""
    g = np.zeros((2, N, N), np.float32)
    g[:, N - 8:, N // 2 - 8:N // 2 + 8] = np.random.default_rng(N).uniform(0.5, 1.0, (2, 8, 16))
    s = 123 - int(np.log2(N))
    assert float(g[0].sum()) * 2.0 ** s * (N - 5) > 3.5e38 > N * float(g[0].sum(1).max()) * 2.0 ** s
    vols = []
    for k in (0, s):
        p = _plan(cp, N, 2, engine=engine)
        p.load_state(g * np.float32(2.0 ** k), 0)
        p.assemble_3d()
        vols.append(p.result(cp.RESULT_VOLUME) / np.float32(2.0 ** k))
        p.close()
    assert np.linalg.norm(vols[1] - vols[0]) < 1e-5 * np.linalg.norm(vols[0])  # the ramps' last bits


def test_refinement_errors(cp):  # noqa: F811
    """One bright voxel: its spectrum is flat, so every term of the error sums
    is 2^120 and their sum is not in FP32."""
    N, Np = 32, 16
    g = np.zeros((Np, N, N), np.float32)
    g[:, N // 2, N // 2] = 1.0
    out = []
    for k in (0, 60):
        p = _plan(cp, N, Np)
        p.load_state(g * np.float32(2.0 ** k), 0)
        p.assemble_3d()
        out.append(p.refine_3d(2))
        p.close()
    np.testing.assert_allclose(out[1], out[0], rtol=1e-6)
    assert out[0][0] > 0.01

"""The warp kernels at the sizes that AUTO sends to them, against the
block-wide engine over the forms a plan can take."""
import itertools

import numpy as np
import pytest

import synth
from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu

# Both sides are FP32 with ~1e-7 log2 N a transform, four transforms a step
# and two steps: 1e-5 leaves a factor of two to five at N = 1024.
TOL = 1e-5


@pytest.mark.parametrize("N", [16, 32, 48, 96, 160, 320, 640, 700, 768])
def test_auto_equals_two_pass(cp, N):  # noqa: F811
    Np = 5
    rng = np.random.default_rng(N)
    q = N // 4
    obj = np.zeros((Np, N, N))
    obj[:, q:N - q, q:N - q] = 1.0 + rng.random((Np, N - 2 * q, N - 2 * q))
    I = np.fft.fftshift(np.abs(np.fft.fft2(obj)) ** 2, axes=(-2, -1)).astype(np.float32)
    S = np.zeros((Np, N, N), np.uint8)
    S[:, q:N - q, q:N - q] = 1
    g0 = (obj + 0.2 * rng.standard_normal(obj.shape)).astype(np.float32)
    y = np.arange(N) - N // 2
    stop = ((y[:, None] ** 2 + y[None, :] ** 2) > 4).astype(np.uint8)
    for mirror, objt, masked, raar in itertools.product((0, 1), repeat=4):
        if N > 320 and mirror != objt:
            continue  # half of the forms at the large sizes
        out = []
        for engine in (cp.ENGINE_TWO_PASS, cp.ENGINE_AUTO):
            p = cp.Plan(cp.make_config(N, Np, n_ei=1, engine=engine, wrap_mode=mirror, blend_target=objt,
                                       update=raar, hio_iters=9 if raar else 0))
            if masked:
                p.load_mask(stop)
            p.load_intensities(I)
            p.load_support(S)
            p.load_state(g0, 0)
            e = p.iterate(2, errors=True)
            out.append((p.result(cp.RESULT_STATE).astype(np.float64), e))
            p.close()
        (a, ea), (b, eb) = out
        rel = np.linalg.norm((a - b).reshape(Np, -1), axis=1) / np.linalg.norm(a.reshape(Np, -1), axis=1)
        assert rel.max() < TOL, (mirror, objt, masked, raar, rel)
        assert np.max(np.abs(ea - eb) / np.maximum(ea, 1e-300)) < 1e-4, (mirror, objt, masked, raar)


@pytest.mark.parametrize("N", [96, 160, 700])
def test_named_engine_refusals_stay(cp, N):  # noqa: F811
    """CPRA_ENGINE_WARP names its list of sizes, whatever AUTO runs."""
    with pytest.raises(cp.CpraError) as e:
        cp.Plan(cp.make_config(N, 2, engine=cp.ENGINE_WARP))
    assert e.value.status == cp.ERR_UNSUPPORTED
    d = synth.make_case("tiny", N=96, Np=2)
    p = cp.Plan(cp.make_config(96, 2))
    p.load_intensities(d["I"], 0, d["thetas"])
    b = cp.Batch([p])
    with pytest.raises(cp.CpraError) as e:
        b.set_persistent(1)
    assert e.value.status == cp.ERR_UNSUPPORTED
    b.close()
    p.close()

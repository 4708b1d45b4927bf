"""The assembly's spectra and grid kernels where their tiles can go wrong,
against the oracle: sizes of every line plan (8, 4, 2 and 1 lines a warp, with
and without idle lanes), planes that do not fill a block, cells that the whole
block sums (more than 32 samples), rows without samples."""
import numpy as np
import pytest

import oracle as O
from test_gpu_parity import TOL, cp  # noqa: F401

pytestmark = pytest.mark.gpu


def _state(N, Np, seed):
    """Iterates off the frame's centre (the mass-centre ramps act) with mass
    in every row, so that the row kz = -N/2 counts."""
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[:N, :N]
    env = np.exp(-((y - 0.55 * N) ** 2 + (x - 0.47 * N) ** 2) / (0.15 * N) ** 2)
    return ((0.2 + env) * rng.standard_normal((Np, N, N)) + env).astype(np.float32)


@pytest.mark.parametrize("N,thetas", [
    (16, np.arange(5) * np.pi / 5),
    (32, np.arange(200) * np.pi / 200),          # heavy cells around the origin
    (48, np.full(40, 0.3)),                      # every cell of one line heavy
    (64, np.array([0.0, 0.4, 0.4, 2.9])),        # rows without samples
    (96, np.arange(7) * np.pi / 7 - 1.0),
    (160, np.arange(3) * np.pi / 3 + 0.1),
    (192, np.arange(2) * np.pi / 2),
    (256, np.array([0.7, 1.9])),
])
@pytest.mark.parametrize("com", [0, 1])
def test_assembly_against_the_oracle(cp, N, thetas, com):  # noqa: F811
    Np = len(thetas)
    g = _state(N, Np, N)
    p = cp.Plan(cp.make_config(N, Np, com_align=com))
    p.load_intensities(np.ones((Np, N, N), np.float32), 0, thetas)
    S = np.ones((N, N), np.uint8)
    S[: N // 8] = 0
    p.load_support(S)
    p.load_state(g, 0)
    vol = np.empty((N, N, N), np.complex64)
    p.assemble_3d(vol)
    p.close()
    ref = O.assemble(g.astype(np.float64), np.broadcast_to(S.astype(bool), g.shape), thetas, com_align=bool(com))
    assert np.linalg.norm(vol - ref) < 0.1 * TOL * np.linalg.norm(ref)
    # the imaginary part is what the unpaired rows and weights leave: small, and right
    assert np.linalg.norm(vol.imag - ref.imag) < 0.1 * TOL * np.linalg.norm(ref)

"""The mirrored 180-degree seam at every kind of size, against the oracle."""
import numpy as np
import pytest

import oracle as O
import synth
from test_gpu_parity import TOL, _one_step, cp  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [16, 32, 48, 64, 96, 160, 192, 256, 320, 384, 512])
def test_mirrored_seam_reads_the_whole_frame(cp, N):  # noqa: F811
    """One coupled RAAR step from an iterate that fills the frame, so that
    column 0 (its own mirror image) counts as much as any other; both angles
    of Np = 2 have a neighbour across the seam."""
    d = synth.make_case("tiny", N=N, Np=2)
    cfg = cp.make_config(N, 2, n_ei=3, wrap_mode=cp.WRAP_MIRROR, update=cp.UPDATE_RAAR,
                         hio_iters=4, er_iters=0)
    g0 = np.random.default_rng(N).standard_normal((2, N, N))
    rel, erel, _ = _one_step(cp, d, cfg, d["support"], g0, 0)
    assert rel.max() < TOL and erel.max() < TOL, (rel, erel)

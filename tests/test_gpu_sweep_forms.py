"""Large groups of Gauss-Seidel guesses run another cluster size or the passes:
every member ends where it ends alone, and the launches are those that
cpra_batch_launches promises."""
import numpy as np
import pytest

import synth
from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,members", [(16, 40), (32, 3), (32, 100), (48, 80), (96, 21), (96, 30), (96, 260), (160, 9), (160, 20),
                                       (320, 14), (320, 24), (320, 32)])
def test_every_member_as_alone(cp, N, members):  # noqa: F811
    import torch
    d = synth.make_case("tiny", N=N, Np=3)
    I = torch.from_numpy(np.asarray(d["I"], np.float32)).cuda()

    def plan(i):
        p = cp.Plan(cp.make_config(N, 3, n_ei=2, seed=i % 3, hio_iters=3, er_iters=1, update=cp.UPDATE_RAAR, sweep=1))
        p.load_intensities(I, 0, d["thetas"])
        p.load_support(d["support"])
        p.iterate(2)
        return p

    alone = []
    for i in range(3):
        p = plan(i)
        p.iterate(2)
        alone.append(p.result(cp.RESULT_STATE))
        p.close()
    group = [plan(i) for i in range(members)]
    b = cp.Batch(group)
    n0 = cp.cpra_launch_count()
    b.iterate(2)
    assert cp.cpra_launch_count() - n0 == b.launches(2)
    for i, p in enumerate(group):
        if i < 6 or i > members - 4 or i % 37 == 0:
            assert np.array_equal(p.result(cp.RESULT_STATE), alone[i % 3])
    b.close()
    for p in group:
        p.close()

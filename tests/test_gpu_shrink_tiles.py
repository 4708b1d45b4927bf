"""The tiled shrink-wrap of the allocation-free entry point where its tiles
can go wrong, against the separate blurs of a plan's shrink-wrap, bit for
bit: sizes that do and do not fill 64 x 32 tiles, one tile a row, supports at
addresses that are not multiples of four, in place, and a Gaussian too wide
for the tile (the separate blurs there too)."""
import numpy as np
import pytest

import synth
from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [64, 96, 160, 192])
@pytest.mark.parametrize("sigma", [0.7, 2.0, 6.0])
def test_tiles_equal_the_separate_blurs(cp, N, sigma):  # noqa: F811
    import torch
    Np = 3
    d = synth.make_case("tiny", N=N, Np=Np)
    plan = cp.Plan(cp.make_config(N, Np, n_ei=2, shrinkwrap_every=1, sw_sigma=sigma, sw_tau=0.2, seed=11,
                                  hio_iters=0, er_iters=4))
    plan.load_intensities(d["I"], 0, d["thetas"])
    plan.load_support(d["support"])
    S0 = torch.from_numpy(np.broadcast_to(d["support"], (Np, N, N)).copy()).cuda()
    g0 = np.random.default_rng(N).standard_normal((Np, N, N)).astype(np.float32)
    g0[1] = 0.0  # a pattern without a maximum keeps its support
    plan.load_state(g0, 1)
    plan.iterate(1)
    g = torch.from_numpy(plan.result(cp.RESULT_STATE)).cuda()
    g[1] = 0.0
    want = plan.result(cp.RESULT_SUPPORT)
    want[1] = d["support"]
    stream = torch.cuda.current_stream().cuda_stream
    for off in (0, 1):  # a support one byte past an aligned address
        room = torch.zeros(Np * N * N + off, dtype=torch.uint8, device="cuda")
        S = room[off:].view(Np, N, N)
        S.copy_(S0)
        S *= 3  # nonzero = in
        out = torch.full((Np, N, N), 7, dtype=torch.uint8, device="cuda")
        cp.cpra_shrinkwrap_static(g, S, out, N, Np, sigma, 0.2, stream)
        assert np.array_equal(out.cpu().numpy()[[0, 2]], want[[0, 2]])
        assert np.array_equal(out.cpu().numpy()[1], want[1])
        cp.cpra_shrinkwrap_static(g, S, S, N, Np, sigma, 0.2, stream)
        assert torch.equal(S, out)
    plan.close()

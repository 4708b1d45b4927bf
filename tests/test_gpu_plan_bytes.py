"""cpra_plan_bytes' second figure against what the first cpra_assemble_3d takes."""
import numpy as np
import pytest

from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Np", [(16, 1), (64, 1), (64, 40), (96, 7), (256, 1), (256, 90)])
def test_assembly_bytes(cp, N, Np):  # noqa: F811
    import torch
    taken = {}

    def alloc(n, ctx):
        t = torch.empty(int(n), dtype=torch.uint8, device="cuda")
        taken[t.data_ptr()] = (t, int(n))
        return t.data_ptr()

    def free(ptr, ctx):
        taken.pop(ptr, None)

    cfg = cp.make_config(N, Np)
    cfg.alloc, cfg.free = cp.binding.ALLOC_FN(alloc), cp.binding.FREE_FN(free)
    promised = cp.cpra_plan_bytes(cfg)[1]
    p = cp.Plan(cfg, stream=torch.cuda.current_stream().cuda_stream, allocator=None)
    p.load_intensities(np.ones((Np, N, N), np.float32), 0, np.arange(Np) * np.pi / Np + 0.1)
    p.iterate(1)  # the step table is the iteration's
    before = sum(n for _, n in taken.values())
    p.assemble_3d()
    used = sum(n for _, n in taken.values()) - before
    p.close()
    # above only by the cells that samples on grid lines do not have (8 bytes
    # each, four a sample at most)
    assert used <= promised <= used + 32 * N * Np

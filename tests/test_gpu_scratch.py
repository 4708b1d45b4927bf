"""Scratch that an allocator cannot give: the assembly, the merge and the
refinement report OUT_OF_MEMORY however far they got, and run once it can."""
import numpy as np
import pytest

import synth
from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu


class Budget:
    """Allocator callbacks that refuse once `left` requests have been granted
    (None: grant all)."""

    def __init__(self, cp):  # noqa: F811
        import torch
        self.left, self.blocks = None, {}

        def alloc(n, ctx):
            if self.left is not None:
                if self.left == 0:
                    return None
                self.left -= 1
            t = torch.empty(int(n), dtype=torch.uint8, device="cuda")
            self.blocks[t.data_ptr()] = t
            return t.data_ptr()

        def free(ptr, ctx):
            self.blocks.pop(ptr, None)

        self.alloc, self.free = cp.binding.ALLOC_FN(alloc), cp.binding.FREE_FN(free)


def _plan(cp, d, seed, budget=None):  # noqa: F811
    import torch
    cfg = cp.make_config(d["N"], d["Np"], seed=seed, hio_iters=0)
    if budget is None:
        p = cp.Plan(cfg)
    else:
        cfg.alloc, cfg.free = budget.alloc, budget.free
        p = cp.Plan(cfg, stream=torch.cuda.current_stream().cuda_stream, allocator=None)
    p.load_intensities(d["I"], 0, d["thetas"])
    p.load_support(d["support"])
    p.iterate(2)
    return p


def _until_granted(cp, budget, call):  # noqa: F811
    """Calls with 0, 1, 2, ... requests granted until one succeeds; the number refused."""
    for k in range(40):
        budget.left = k
        try:
            call()
            return k
        except cp.CpraError as e:
            assert e.status == cp.ERR_OUT_OF_MEMORY
        finally:
            budget.left = None
    raise AssertionError("never granted")


def test_scratch_running_out_leaves_the_plan_usable(cp):  # noqa: F811
    d = synth.make_case("tiny", N=64, Np=6)
    b = Budget(cp)
    p, q = _plan(cp, d, 1, b), _plan(cp, d, 1)
    other = _plan(cp, d, 2)

    def same():
        x, y = p.result(cp.RESULT_VOLUME), q.result(cp.RESULT_VOLUME)
        assert np.linalg.norm(x - y) < 1e-6 * np.linalg.norm(y)  # FP64 atomics order the mass centres' last bits

    assert _until_granted(cp, b, p.assemble_3d) > 1
    q.assemble_3d()
    same()
    assert _until_granted(cp, b, lambda: p.refine_3d(2)) > 1
    q.refine_3d(2)
    same()
    assert _until_granted(cp, b, lambda: p.refine_3d(3)) == 1  # longer error sums alone
    q.refine_3d(3)
    same()
    out = []
    for dst in (p, q):
        prtf = np.empty((d["Np"], d["N"] // 2), np.float32)
        call = lambda: cp.cpra_merge([dst, other], 2, 0, dst, prtf)  # noqa: B023, E731
        if dst is p:
            assert _until_granted(cp, b, call) > 1
        else:
            call()
        out.append(prtf)
    same()
    np.testing.assert_allclose(out[0], out[1], rtol=1e-5)
    for x in (p, q, other):
        x.close()
    assert not b.blocks

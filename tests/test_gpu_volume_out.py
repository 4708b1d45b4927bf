"""cpra_assemble_3d into the caller's device memory: the last kernel writes it,
so a buffer that a copy would have refused is refused before any launch."""
import numpy as np
import pytest

from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu


def test_a_short_device_buffer_is_refused(cp):  # noqa: F811
    import torch
    N = 128
    p = cp.Plan(cp.make_config(N, 2))
    p.load_intensities(np.ones((2, N, N), np.float32), 0, np.array([0.1, 1.0]))
    p.load_state(np.random.default_rng(0).random((2, N, N)).astype(np.float32), 0)
    p.assemble_3d()
    want = p.result(cp.RESULT_VOLUME)
    short = torch.empty(1000, dtype=torch.complex64, device="cuda")  # in a segment of 2 MB; the volume has 16
    n0 = cp.cpra_launch_count()
    with pytest.raises(cp.CpraError) as e:
        p.assemble_3d(short)
    assert e.value.status == cp.ERR_INVALID_ARG and cp.cpra_launch_count() == n0
    # and what was accepted still is: a whole buffer, the tail of a larger one, unaligned device memory, host memory
    big = torch.empty(3 * N ** 3, dtype=torch.complex64, device="cuda")
    odd = torch.empty(2 * N ** 3 + 1, dtype=torch.float32, device="cuda")
    host = np.empty((N, N, N), np.complex64)
    for out in (big[:N ** 3], big[2 * N ** 3:], odd[1:], host):
        p.assemble_3d(out)
        got = out if out is host else torch.view_as_real(out).cpu().numpy() if out.is_complex() else out.cpu().numpy()
        got = np.ascontiguousarray(got).view(np.float32).reshape(N, N, N, 2)
        np.testing.assert_allclose(got, want.view(np.float32).reshape(N, N, N, 2), rtol=0, atol=1e-5 * np.abs(want).max())
    p.close()

"""Inputs that torch is still computing when a call starts: the call waits for them (a context works on a
stream of its own)."""
import numpy as np
import pytest

from paper_1909_10690_gb300 import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["hard", "parzen"])
def test_device_inputs_still_being_computed(cuda_lib, kernel):
    import torch

    f, m = phantoms.ellipsoid_pair(shape=(40, 40, 40), seed=75)
    T = phantoms.random_transforms(3, seed=76, t_mm=2, r_deg=5, s_range=(0.95, 1.05))
    want = cuda_lib.Context(f, m, bins=32, kernel=kernel).eval(T, [1.0])
    fd, md, Td = (torch.from_numpy(a).cuda() for a in (f, m, T))
    busy = torch.randn(4096, 4096, device="cuda")
    late = [torch.zeros_like(x) for x in (fd, md, Td)]
    torch.cuda.synchronize()
    for _ in range(30):  # tens of milliseconds of queued work before the inputs are written
        busy = (busy @ busy).clamp_(-1, 1)
    late[0].copy_(fd)
    late[1].copy_(md)
    ctx = cuda_lib.Context(late[0], late[1], bins=32, kernel=kernel)
    for _ in range(30):
        busy = (busy @ busy).clamp_(-1, 1)
    late[2].copy_(Td)
    np.testing.assert_array_equal(ctx.eval(late[2], [1.0]).cpu().numpy(), want)

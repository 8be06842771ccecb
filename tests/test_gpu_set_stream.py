"""Switching a context's stream: what the old stream still holds for the context is waited for, and nothing else."""
import numpy as np
import pytest

from paper_1909_10690_gb300 import phantoms

pytestmark = pytest.mark.gpu


def _keep_busy(torch, x, n):
    for _ in range(n):
        x = (x @ x).clamp_(-1, 1)
    return x


def test_entropy_table_of_a_failed_call(cuda_lib):
    """The first of two tables is queued behind other work on A, the second's allocation fails; the next call
    reads the first on B."""
    import torch

    f, m = phantoms.head_pair(shape=(24, 26, 28), spacing=(1, 1, 1), seed=100)
    prm = phantoms.random_transforms(3, seed=101, t_mm=3, r_deg=8, s_range=(0.95, 1.05))
    kw = dict(bins=64, fixed_depth=12, moving_depth=12)
    want = cuda_lib.Context(f, m, **kw).eval(prm, [1.5])
    ctx = cuda_lib.Context(f, m, **kw)
    A, B = torch.cuda.Stream(), torch.cuda.Stream()
    ctx.set_stream(A)
    x = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(A):
        x = _keep_busy(torch, x, 30)
    lib = cuda_lib.load()
    try:
        lib.mi_fault_alloc(1)
        with pytest.raises(cuda_lib.MIError) as e:
            ctx.eval(prm, [1.5, 2.5])
        assert e.value.status == cuda_lib.MI_ENOMEM
    finally:
        lib.mi_fault_alloc(-1)
    ctx.set_stream(B)
    np.testing.assert_array_equal(ctx.eval(prm, [1.5]), want)
    torch.cuda.synchronize()


@pytest.mark.parametrize("call", ["resample", "eval"])
def test_nothing_is_waited_for_after_a_finished_call(cuda_lib, call):
    import torch

    f, m = phantoms.head_pair(shape=(24, 26, 28), spacing=(1, 1, 1), seed=102)
    ctx = cuda_lib.Context(f, m, bins=64, fixed_depth=12, moving_depth=12)
    prm = phantoms.identity_params(1)
    if call == "resample":
        ctx.resample(ctx.affine(prm)[1][0])
    else:
        ctx.eval(prm)
    x = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    x = _keep_busy(torch, x, 100)
    end = torch.cuda.Event()
    end.record()
    ctx.set_stream(torch.cuda.Stream())
    assert not end.query()
    torch.cuda.synchronize()

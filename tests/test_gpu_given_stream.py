"""A context that was given a stream works in that stream's order and beside the other streams' work."""
import numpy as np
import pytest

from paper_1909_10690_gb300 import phantoms

pytestmark = pytest.mark.gpu

QS = [1.0, 1.5]


def _keep_busy(torch, x, n):
    for _ in range(n):
        x = (x @ x).clamp_(-1, 1)
    return x


@pytest.mark.parametrize("call", ["eval", "eval_q16", "batch_eval", "grad", "hist"])
def test_other_streams_are_not_waited_for(cuda_lib, call):
    """Inputs made on S, a call on S, while the current stream has most of a second of work queued: the call's
    results are there before that work ends, and right."""
    import torch

    f, m = phantoms.ellipsoid_pair(shape=(40, 40, 40), seed=92)
    prm = phantoms.random_transforms(3, seed=93, t_mm=2, r_deg=5, s_range=(0.95, 1.05))
    parzen = call == "grad"
    pairs = [dict(fixed=f, moving=m, bins=32)] * 2 if call == "batch_eval" else None
    make = lambda: (cuda_lib.Context(pairs=pairs) if pairs else  # noqa: E731
                    cuda_lib.Context(f, m, bins=32, kernel="parzen" if parzen else "hard"))
    ctx = make()

    def run(c, T, P, A):
        if call == "eval":
            return c.eval(T, QS, with_entropies=True)
        if call == "eval_q16":
            return c.eval_q16(A, QS, with_entropies=True)
        if call == "batch_eval":
            return c.batch_eval(P, T, QS)
        return c.grad(T, QS) if parzen else c.hist(transforms=T)

    S = torch.cuda.Stream()
    ctx.set_stream(S)
    host = (prm, np.array([1, 0, 1], np.int32), ctx.affine(prm)[1])
    want = run(make(), *host)
    with torch.cuda.stream(S):
        T, P, A = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in host)
    T = T.double() if call == "eval" else T  # converted by the call
    torch.cuda.synchronize()
    run(ctx, T, P, A)  # allocations are made before the timed call
    x = _keep_busy(torch, torch.randn(4096, 4096, device="cuda"), 3)
    torch.cuda.synchronize()
    x = _keep_busy(torch, x, 300)
    end = torch.cuda.Event()
    end.record()
    got = run(ctx, T, P, A)
    assert not end.query()
    for a, b in zip(got if isinstance(got, tuple) else (got,), want if isinstance(want, tuple) else (want,)):
        np.testing.assert_allclose(a.cpu().numpy() if torch.is_tensor(a) else a, b, rtol=1e-12, atol=1e-13)
    torch.cuda.synchronize()


@pytest.mark.parametrize("raw", [False, True])
def test_inputs_still_being_computed_on_the_given_stream(cuda_lib, raw):
    import torch

    f, m = phantoms.ellipsoid_pair(shape=(40, 40, 40), seed=94)
    prm = phantoms.random_transforms(3, seed=95, t_mm=2, r_deg=5, s_range=(0.95, 1.05))
    ctx = cuda_lib.Context(f, m, bins=32)
    want = ctx.eval(prm, QS)
    S = torch.cuda.Stream()
    ctx.set_stream(S.cuda_stream if raw else S)
    Td = torch.from_numpy(prm).cuda()
    late = torch.zeros_like(Td)
    x = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(S):
        x = _keep_busy(torch, x, 30)
        late.copy_(Td)
    np.testing.assert_array_equal(ctx.eval(late, QS).cpu().numpy(), want)
    ctx.set_stream(None)
    np.testing.assert_array_equal(ctx.eval(late, QS).cpu().numpy(), want)


def test_outputs_outlive_the_readers_queued_behind_them(cuda_lib):
    """An output read by work that waits on the caller's stream, then dropped: its memory is not written by the
    next call on the given stream."""
    import torch

    f, m = phantoms.ellipsoid_pair(shape=(40, 40, 40), seed=96)
    prm = phantoms.random_transforms(600, seed=97, t_mm=4, r_deg=15, s_range=(0.9, 1.1))
    ctx = cuda_lib.Context(f, m, bins=32)
    want = ctx.eval(prm[:300], QS)
    S = torch.cuda.Stream()
    ctx.set_stream(S)
    with torch.cuda.stream(S):
        a, b = torch.from_numpy(prm[:300]).cuda(), torch.from_numpy(prm[300:]).cuda()
    torch.cuda.synchronize()
    ctx.eval(b, QS)
    x = _keep_busy(torch, torch.randn(4096, 4096, device="cuda"), 100)
    out = ctx.eval(a, QS)
    kept = out.clone()  # runs behind the queued work
    del out
    for _ in range(3):
        ctx.eval(b, QS)
    np.testing.assert_array_equal(kept.cpu().numpy(), want)


def test_gradient_function_is_an_operator_of_the_current_stream(cuda_lib):
    """theta written late on the current stream, a context on another one."""
    import torch

    f, m = phantoms.ellipsoid_pair(shape=(32, 32, 32), seed=98)
    prm = phantoms.random_transforms(2, seed=99, t_mm=2, r_deg=5, s_range=(0.95, 1.05))
    ctx = cuda_lib.Context(f, m, bins=32, kernel="parzen")
    want, _ = ctx.grad(prm, QS)
    ctx.set_stream(torch.cuda.Stream())
    theta = torch.zeros(prm.shape, dtype=torch.float64, device="cuda", requires_grad=True)
    Td = torch.from_numpy(prm).cuda()
    _keep_busy(torch, torch.randn(4096, 4096, device="cuda"), 30)
    with torch.no_grad():
        theta.copy_(Td)
    got = cuda_lib.mi_function().apply(theta, ctx, QS)
    np.testing.assert_array_equal(got.detach().cpu().numpy(), want)
    got.sum().backward()
    assert torch.isfinite(theta.grad).all()

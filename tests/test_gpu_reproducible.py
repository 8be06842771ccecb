"""Repeated calls of one context agree bit for bit, with many cells beyond the entropy table (their terms are
listed and summed side by side, in an order that must not depend on which warp came first)."""
import numpy as np
import pytest

from paper_1909_10690_gb300 import phantoms

pytestmark = pytest.mark.gpu

QS = [0.5, 1.0, 1.5, 2.0, 3.0, 2.5]


@pytest.mark.parametrize("bins,n,path,size", [
    (6, 8, "batched", 160),    # 36 large cells a transform, reduced in place
    (128, 90, "plain", 160),   # head-like: through slots, four parts each
    (64, 320, "plain", 128),   # one part a slot
    (18, 2, "batched", 288),   # more large cells than the list holds
])
def test_repeated_calls_bit_for_bit(cuda_lib, bins, n, path, size):
    if bins in (6, 18):
        rng = np.random.default_rng(110)
        f, m = (rng.integers(0, 256, (size, size, size), dtype=np.uint8) for _ in range(2))
        ctx = cuda_lib.Context(f, m, bins=bins, path=path, autotune=False)
    else:
        f, m = phantoms.head_pair(shape=(size, size, size), spacing=(1, 1, 1), seed=111)
        ctx = cuda_lib.Context(f, m, bins=bins, fixed_depth=12, moving_depth=12, path=path, autotune=False)
    prm = phantoms.random_transforms(n, seed=112, t_mm=2, r_deg=3, s_range=(0.98, 1.02))
    if bins in (6, 18):
        prm[:] = phantoms.identity_params(1)
    mi, h, _ = ctx.eval(prm, QS, with_entropies=True)
    if bins in (6, 18):
        assert (ctx.hist(transforms=prm[:1]) >= 65536).sum() == bins * bins
    for _ in range(15):
        mi2, h2, _ = ctx.eval(prm, QS, with_entropies=True)
        np.testing.assert_array_equal(mi2, mi)
        np.testing.assert_array_equal(h2, h)

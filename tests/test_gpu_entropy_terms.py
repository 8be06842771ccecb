"""The terms behind the entropies (table and series, counted cells, listed large counts) against exact counts.

Tolerances: a term v ln v or v^q of the table and series is within 4.1e-16 of its value, so H = (N ln N - S) / N
is within 2 x ln N x 4.1e-16 < 2e-14 for q = 1 (N < 2^21), and (1 - S / N^q) / (q - 1) within
(8.2e-16 + 3 roundings) / |q - 1| < 4e-15 for |q - 1| >= 1/2.
"""
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_1909_10690_gb300 import phantoms

pytestmark = pytest.mark.gpu


def _entropy(counts, q):
    """60-digit entropy of whole counts."""
    getcontext().prec = 60
    n, q = Decimal(sum(counts)), Decimal(float(np.float32(q)))
    if q == 1:
        return float(n.ln() - sum(Decimal(c) * Decimal(c).ln() for c in counts) / n)
    return float((1 - sum((q * (Decimal(c) / n).ln()).exp() for c in counts)) / (q - 1))


@pytest.mark.parametrize("path", ["plain", "batched", "noalloc"])
def test_series_of_large_counts(cuda_lib, path):
    """Two cells of 1114111 and 16385 voxels: the first is 2^5 x 34815 + 31 and 2^13 x 135 + 8191, where the
    series' argument is nearly the largest (2.8e-5 beyond 16 bits, 0.0074 beyond 8), the total 2^13 x 138, where it is 0.
    At q = 7 the series without its third term would be off by 1e-13 in H, the allocation-free call's (8 terms)
    without its sixth by as much at q = 6.5."""
    import torch

    shape, big = (96, 92, 128), 1114111
    f = np.zeros(shape, np.uint8)
    f.reshape(-1)[big:] = 255
    small = f.size - big
    qs = [1.0, 1.5, 6.5, 7.0]
    want = np.array([_entropy([big, small], q) for q in qs])
    tol = np.array([2e-14, 4e-15, 4e-15, 4e-15])
    prm = phantoms.identity_params(1)
    if path == "noalloc":
        d = torch.from_numpy(f).cuda()
        got = cuda_lib.eval_noalloc(d, d, 2, prm[0], qs)
        assert np.all(np.abs(got - want) <= tol), got - want
        return
    mi, h, cnt = cuda_lib.Context(f, f, bins=2, path=path).eval(prm, qs, with_entropies=True)
    assert cnt[0] == f.size
    assert np.all(np.abs(h[0] - want[:, None]) <= tol[:, None]), h[0] - want[:, None]
    assert np.all(np.abs(mi[0] - want) <= tol), mi[0] - want


def test_more_large_counts_than_the_list_holds(cuda_lib):
    """324 cells of 71 000 voxels and more, where a CTA lists 255 of them, and six q, so that a second pass over
    the cells takes the ones the first took on the way."""
    rng = np.random.default_rng(109)
    f, m = (rng.integers(0, 256, (288, 288, 288), dtype=np.uint8) for _ in range(2))
    bins, qs = 18, [0.5, 1.0, 1.5, 2.0, 3.0, 7.0]
    ctx = cuda_lib.Context(f, m, bins=bins, path="batched")
    prm = phantoms.identity_params(1)
    H = ctx.hist(transforms=prm)[0].astype(np.int64)
    fb, mb = ((v.reshape(-1).astype(np.int64) * bins) >> 8 for v in (f, m))
    np.testing.assert_array_equal(H, np.bincount(fb * bins + mb, minlength=bins * bins).reshape(bins, bins))
    assert (H >= 65536).sum() > 255
    mi, h, cnt = ctx.eval(prm, qs, with_entropies=True)
    assert cnt[0] == f.size
    for iq, q in enumerate(qs):
        want = [_entropy([int(c) for c in line], q) for line in (H.sum(1), H.sum(0), H.reshape(-1))]
        # up to 342 terms, whose errors are independent, and their sum: a hundredfold of one term's
        assert np.all(np.abs(h[0, iq] - want) <= 1e-12 * np.maximum(np.abs(want), 1.0)), (q, h[0, iq] - want)
        assert abs(mi[0, iq] - (want[0] + want[1] - want[2])) <= 3e-12 * max(1.0, *np.abs(want)), q

"""Bin counts and plane counts at which a CTA's shared memory comes near the 227 KB it can have.

The gather variants keep 8 bytes per moving plane behind their 32-bit counters, and the entropy reduction's
table of small counts (4 KB) is optional.  Tolerance: the hard path's, 1e-6 max(|MI|, H_FM); counts are whole
numbers and equal.
"""
import numpy as np
import pytest

import oracle
from paper_1909_10690_gb300 import phantoms

pytestmark = pytest.mark.gpu


def _compare(cuda_lib, bins, planes, ns):
    rng = np.random.default_rng(90)
    f = rng.integers(0, 4096, (40, 6, 9), dtype=np.uint16)
    m = rng.integers(0, 4096, (planes, 7, 10), dtype=np.uint16)
    prm = phantoms.random_transforms(max(ns), seed=91, t_mm=1, r_deg=5, s_range=(0.9, 1.1))
    qs = [1.0, 2.0]
    mi_o, h_o, cnt_o = oracle.mi_eval(f, m, bins, prm, qs, fixed_depth=12, moving_depth=12, nthreads=8)
    ok = cnt_o > 0
    for kw in (dict(hist_variant=cuda_lib.HV_U32_GATHER), {}):
        ctx = cuda_lib.Context(f, m, bins=bins, fixed_depth=12, moving_depth=12, **kw)
        for n in ns:  # above the SM count: every candidate is timed
            mi, _, cnt = ctx.eval(prm[:n], qs, with_entropies=True)
            np.testing.assert_array_equal(cnt, cnt_o[:n])
            g = ok[:n]
            assert np.all(np.abs(mi[g] - mi_o[:n][g]) <= 1e-6 * np.maximum(np.abs(mi_o[:n][g]), h_o[:n][g][..., 2]) + 1e-12)
        if kw:
            assert ctx.selected_variant(max(ns)) == cuda_lib.HV_U32_GATHER


@pytest.mark.parametrize("bins,planes", [(236, 222), (236, 300), (236, 511), (235, 470)])
def test_no_room_for_the_table_behind_the_plane_offsets(cuda_lib, bins, planes):
    """The counters leave 4 KB for the table, the counters and the plane offsets do not."""
    _compare(cuda_lib, bins, planes, (160,))

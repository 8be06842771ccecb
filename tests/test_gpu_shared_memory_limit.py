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


@pytest.mark.parametrize("bins,planes", [(236, 214), (236, 218), (236, 221), (238, 248), (238, 252), (238, 255),
                                         (239, 12), (239, 15)])
def test_static_variables_beside_the_largest_layouts(cuda_lib, bins, planes):
    """0 to 56 bytes less than 227 KB with the table (236) or without it: the kernel's static variables do not
    fit beside that, so the table is left out, or the variant, and no error is left for a later call."""
    rng = np.random.default_rng(92)
    if bins == 236:
        _compare(cuda_lib, bins, planes, (1, 160))
        return
    f = rng.integers(0, 4096, (40, 6, 9), dtype=np.uint16)
    m = rng.integers(0, 4096, (planes, 7, 10), dtype=np.uint16)
    prm = phantoms.random_transforms(160, seed=93, t_mm=1, r_deg=5, s_range=(0.9, 1.1))
    want, h, cnt_o = oracle.mi_eval(f, m, bins, prm, [1.0], fixed_depth=12, moving_depth=12, nthreads=8)
    for n in (1, 160):
        ctx = cuda_lib.Context(f, m, bins=bins, fixed_depth=12, moving_depth=12)
        got, _, cnt = ctx.eval(prm[:n], [1.0], with_entropies=True)
        np.testing.assert_array_equal(cnt, cnt_o[:n])
        ok = cnt > 0
        assert np.all(np.abs(got[ok] - want[:n][ok]) <= 1e-6 * np.maximum(np.abs(want[:n][ok]), h[:n][ok][..., 2]) + 1e-12)
    with pytest.raises(cuda_lib.MIError) as e:
        cuda_lib.Context(f, m, bins=bins, fixed_depth=12, moving_depth=12, hist_variant=cuda_lib.HV_U32_GATHER).eval(prm[:1])
    assert e.value.status == cuda_lib.MI_EUNSUPPORTED
    cuda_lib.Context(f, m, bins=32, fixed_depth=12, moving_depth=12).eval(prm[:1])

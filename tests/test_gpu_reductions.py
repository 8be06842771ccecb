"""The reductions after the voxel kernels, at the sizes where their splits change, against the oracle.

Tolerances are those of the paths they end: hard MI within 1e-6 max(|MI|, H_FM), Parzen MI within
1e-6 max(|MI|, 1) and gradients within 1e-4 of the largest component (FP32 weights and moments).
"""
import numpy as np
import pytest

import oracle
from paper_1909_10690_gb300 import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,bins,n", [((3, 5, 40), 8, 1), ((20, 30, 24), 17, 1), ((40, 40, 33), 128, 1),
                                          ((20, 30, 24), 96, 40)])
def test_parzen_marginals_and_moment_sums(cuda_lib, shape, bins, n):
    """Few and many adjoint parts per transform (one warp's rows up to every SM), column slices that
    do and do not divide the threads, and every q at once."""
    f, m = phantoms.head_pair(shape=shape, spacing=(1, 1, 1), seed=60, dtype=np.float32)
    qs = [1.0, 0.7, 1.3, 2.0, 3.0]
    prm = phantoms.random_transforms(n, seed=61, t_mm=1, r_deg=4, s_range=(0.97, 1.03))
    mi, g = cuda_lib.Context(f, m, bins=bins, kernel="parzen").grad(prm, qs)
    for t in range(0, n, max(1, n // 4)):
        aff, J = oracle.affine(prm[t], f.shape, (1, 1, 1), m.shape, (1, 1, 1), with_jacobian=True)
        mi_o, g_o, _ = oracle.parzen(f, m, aff, bins, qs, daff=J)
        assert np.all(np.abs(mi[t] - mi_o) <= 1e-6 * np.maximum(np.abs(mi_o), 1.0))
        for iq in range(len(qs)):
            assert np.abs(g[t, iq] - g_o[iq]).max() <= 1e-4 * np.abs(g_o[iq]).max()

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
    # (q < 1 is left out: on 13 000 voxels over 96 bins W = P^(q-1) of the cells that hold only B-spline
    # tails follows the FP32 weights' error, 1.7e-4 of the gradient at q = 0.7 whatever sums it)
    qs = [1.0, 1.3, 2.0, 3.0, 4.0]
    prm = phantoms.random_transforms(n, seed=61, t_mm=1, r_deg=4, s_range=(0.97, 1.03))
    mi, g = cuda_lib.Context(f, m, bins=bins, kernel="parzen").grad(prm, qs)
    for t in range(0, n, max(1, n // 4)):
        aff, J = oracle.affine(prm[t], f.shape, (1, 1, 1), m.shape, (1, 1, 1), with_jacobian=True)
        mi_o, g_o, _ = oracle.parzen(f, m, aff, bins, qs, daff=J)
        assert np.all(np.abs(mi[t] - mi_o) <= 1e-6 * np.maximum(np.abs(mi_o), 1.0))
        for iq in range(len(qs)):
            assert np.abs(g[t, iq] - g_o[iq]).max() <= 1e-4 * np.abs(g_o[iq]).max()


@pytest.mark.parametrize("n,bins,path", [(1, 32, "auto"), (2, 256, "auto"), (75, 128, "auto"), (151, 64, "auto"),
                                         (153, 64, "auto"), (330, 100, "auto"), (1, 32, "plain"), (330, 100, "plain")])
def test_split_transforms(cuda_lib, n, bins, path):
    """Transforms cut into parts over the CTAs: from one transform over all of them to a split tail behind
    whole ones, rows that do not divide into the parts, an empty overlap among them, nine-tenths of the
    cells holding small counts and some above the count-of-counts table; repeated (graph) calls agree."""
    f, m = phantoms.head_pair(shape=(45, 38, 52), spacing=(1, 1, 1), seed=62)
    prm = phantoms.random_transforms(n, seed=63, t_mm=4, r_deg=12, s_range=(0.9, 1.1))
    if n > 2:
        prm[n // 2, 0] = 500.0  # no overlap
    qs = [0.5, 1.0, 1.5, 2.0, 3.0]
    ctx = cuda_lib.Context(f, m, bins=bins, fixed_depth=12, moving_depth=12, path=path)
    mi_o, h_o, cnt_o = oracle.mi_eval(f, m, bins, prm, qs, fixed_depth=12, moving_depth=12, nthreads=8)
    ok = cnt_o > 0
    for _ in range(3):
        mi, h, cnt = ctx.eval(prm, qs, with_entropies=True)
        np.testing.assert_array_equal(cnt, cnt_o)
        assert np.all(np.isnan(mi[~ok]))
        assert np.all(np.abs(mi[ok] - mi_o[ok]) <= 1e-6 * np.maximum(np.abs(mi_o[ok]), h_o[ok][..., 2]) + 1e-12)
        assert np.all(np.abs(h[ok] - h_o[ok]) <= 1e-9 * np.maximum(np.abs(h_o[ok]), 1.0))
    T = ctx.hist(transforms=prm[:1])
    q16 = oracle.affine_q16(oracle.affine(prm[0], f.shape, (1, 1, 1), m.shape, (1, 1, 1)))
    ho, _ = oracle.joint_hist(f, m, q16, bins, fixed_depth=12, moving_depth=12)
    np.testing.assert_array_equal(T[0], ho.astype(np.uint32))


@pytest.mark.parametrize("fraction", [0.0, 0.2])
def test_split_pairs_of_unequal_size(cuda_lib, fraction):
    """A few transforms on pairs of very different sizes and bins: the large ones are cut, the small are not."""
    specs = [((60, 50, 70), np.uint16, 12, 128), ((9, 12, 20), np.uint8, 8, 32), ((30, 44, 38), np.uint8, 8, 64)]
    pairs, vols = [], []
    for i, (shape, dt, depth, bins) in enumerate(specs):
        f, m = phantoms.head_pair(shape=shape, spacing=(1, 1, 1), seed=64 + i, depth=depth, dtype=dt)
        vols.append((f, m, depth, bins))
        pairs.append(dict(fixed=f, moving=m, bins=bins, fixed_depth=depth, moving_depth=depth))
    ctx = cuda_lib.Context(pairs=pairs, sample_fraction=fraction, sample_seed=5)
    whole = [cuda_lib.Context(**p, sample_fraction=fraction, sample_seed=5, path="batched") for p in pairs]
    po = np.array([1, 0, 2, 0, 1, 1, 2], np.int32)
    prm = phantoms.random_transforms(len(po), seed=67, t_mm=2, r_deg=8, s_range=(0.95, 1.05))
    qs = [1.0, 2.0]
    mi, h, cnt = ctx.batch_eval(po, prm, qs, with_entropies=True)
    for t, p in enumerate(po):
        want, hw, cw = whole[p].eval(prm[t:t + 1], qs, with_entropies=True)
        assert cnt[t] == cw[0]
        np.testing.assert_allclose(mi[t], want[0], rtol=0, atol=1e-11)
        np.testing.assert_allclose(h[t], hw[0], rtol=0, atol=1e-11)


@pytest.mark.parametrize("shape,dtype,depth,bins", [((2, 2, 2), np.uint8, 8, 2), ((5, 7, 33), np.uint16, 16, 256),
                                                    ((40, 44, 52), np.uint16, 12, 160), ((40, 44, 52), np.uint16, 12, 161),
                                                    ((64, 64, 64), np.uint8, 7, 32)])
def test_noalloc_rows_counters_and_terms(cuda_lib, shape, dtype, depth, bins):
    """The allocation-free call against the oracle: fewer rows than warps and many, 32- and 16-bit counters
    at the bin count where they change, a depth below the type's, counts below 256, in the series' range
    and (one cell of a constant pair) at the volume's size, q above the series' range."""
    import torch

    rng = np.random.default_rng(70)
    if min(shape) < 8:
        f, m = (rng.integers(0, 1 << depth, shape).astype(dtype) for _ in range(2))
    else:
        f, m = (v.astype(dtype) for v in phantoms.head_pair(shape=shape, spacing=(1, 1, 1), seed=71, depth=depth, dtype=dtype))
    qs = [1.0, 0.5, 1.5, 2.0, 7.0, 8.5]
    prm = np.concatenate([phantoms.identity_params(1), phantoms.random_transforms(2, seed=72, t_mm=0.5, r_deg=6, s_range=(0.95, 1.05))])
    for a, b in ((f, m), (np.zeros_like(f), np.zeros_like(m))):
        mi_o, h_o, cnt = oracle.mi_eval(a, b, bins, prm, qs, fixed_depth=depth, moving_depth=depth, nthreads=8)
        ad, bd = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        for t in range(len(prm)):
            if cnt[t] == 0:
                continue
            got = cuda_lib.eval_noalloc(ad, bd, bins, prm[t], qs, fixed_depth=depth, moving_depth=depth)
            assert np.all(np.abs(got - mi_o[t]) <= 1e-6 * np.maximum(np.abs(mi_o[t]), h_o[t, :, 2]) + 1e-12)


@pytest.mark.parametrize("bins,nq,sampled", [(8, 1, False), (64, 2, False), (128, 3, False), (96, 4, False),
                                             (97, 4, False), (33, 7, False), (64, 3, True)])
def test_adjoint_tables(cuda_lib, bins, nq, sampled):
    """Paired and single q tables in shared and in global memory (four q from 97 bins on), an odd number of
    fixed rows, saturated intensities (the last moving bin, whose last tap is outside the table), random
    sampling, and a second pair with fewer bins in the same call."""
    rng = np.random.default_rng(78)
    f, m = phantoms.head_pair(shape=(27, 31, 37), spacing=(1, 1, 1), seed=77, dtype=np.float32)
    f[rng.random(f.shape) < 0.05] = 1.0
    m[10:14, 8:20, 5:30] = 1.0
    qs = [1.0, 1.3, 2.0, 3.0, 4.0, 1.5, 2.5][:nq]
    prm = phantoms.random_transforms(3, seed=79, t_mm=6, r_deg=15, s_range=(0.9, 1.1))
    kw = dict(kernel="parzen", sample_fraction=0.3 if sampled else 0.0, sample_seed=4)
    thr = oracle.sample_threshold(0.3)
    keep = np.array([oracle.sampled(x, 4, thr) for x in range(f.size)]).reshape(f.shape) if sampled else None
    _, g = cuda_lib.Context(f, m, bins=bins, **kw).grad(prm, qs)
    _, gm = cuda_lib.Context(pairs=[dict(fixed=f, moving=m, bins=b) for b in (bins, 16)], **kw).batch_grad(
        np.array([0, 1, 0], np.int32), prm, qs)
    for t in range(3):
        aff, J = oracle.affine(prm[t], f.shape, (1, 1, 1), m.shape, (1, 1, 1), with_jacobian=True)
        mask = keep & oracle.overlap_mask(f.shape, m.shape, aff) if sampled else None
        for got, b in ((g[t], bins), (gm[t], (bins, 16, bins)[t])):
            _, want, _ = oracle.parzen(f, m, aff, b, qs, daff=J, mask=mask)
            for iq in range(nq):
                assert np.abs(got[iq] - want[iq]).max() <= 1e-4 * np.abs(want[iq]).max(), (t, b, iq)


def test_parzen_row_clipping(cuda_lib):
    """Overlap counts and MI where a row's interval comes from very small, zero, negative and very large
    steps, on a dark, a bright and a full-range volume."""
    rng = np.random.default_rng(81)
    base = np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0], np.float32)
    prm = np.repeat(base[None], 8, axis=0)
    prm[1, [0, 3]] = (-1.0, 0.25)
    prm[2, 0] = 0.0
    prm[3, [0, 5]] = (1e-7, -1e-7)
    prm[4, [0, 7]] = (37.0, 2.5)
    prm[5, 0] = -3e-10
    prm[6, [0, 4, 8]] = (0.7, 0.7, -0.7)
    prm[7, [0, 10]] = (-250.0, 0.5)
    for shape, lo, hi, bins in (((9, 17, 70), 0.0, 0.1, 8), ((9, 17, 70), 0.93, 1.0, 128), ((12, 9, 33), 0.0, 1.0, 64)):
        f, m = (rng.uniform(lo, hi, shape).astype(np.float32) for _ in range(2))
        f[:, :, :9] = rng.uniform(0, 1)
        ctx = cuda_lib.Context(f, m, bins=bins, kernel="parzen", transform="affine")
        mi, _, cnt = ctx.eval(prm, [1.0, 2.0], with_entropies=True)
        for t in range(len(prm)):
            aff = oracle.affine(prm[t], f.shape, (1, 1, 1), m.shape, (1, 1, 1), transform="affine")
            want, _, n = oracle.parzen(f, m, aff, bins, [1.0, 2.0])
            assert cnt[t] == n, (t, cnt[t], n)
            if n > 1:
                assert np.all(np.abs(mi[t] - want) <= 1e-6 * np.maximum(np.abs(want), 1.0)), (t, mi[t], want)


@pytest.mark.parametrize("variant", ["HV_U32_QUAD", "HV_U16_QUAD", "HV_ROWS_QUAD", "HV_U32_GATHER", "HV_U16_GATHER", "HV_ROWS_GATHER"])
@pytest.mark.parametrize("rows", [1, 2, 4, 32])
def test_byte_volumes_in_paired_lanes(cuda_lib, variant, rows):
    """8-bit moving volumes at full range (0 and 255 beside each other: the largest 16-bit lane sums), through
    both texture fetches and every walk, whole and split: histograms equal the oracle's, also in a
    context that holds a 16-bit pair beside them; 31 fixed rows a slice leave every group ragged."""
    rng = np.random.default_rng(83)
    f = rng.integers(0, 256, (9, 31, 45), dtype=np.uint8)
    m = np.where(rng.random((11, 27, 40)) < 0.5, 0, 255).astype(np.uint8)
    m[:5] = rng.integers(0, 256, (5, 27, 40), dtype=np.uint8)
    kw = dict(hist_variant=getattr(cuda_lib, variant), tile_rows=rows)
    prm = phantoms.random_transforms(4, seed=84, t_mm=3, r_deg=20, s_range=(0.8, 1.2))
    ctx = cuda_lib.Context(f, m, bins=64, **kw)
    f16, m16 = phantoms.head_pair(shape=(12, 14, 20), spacing=(1, 1, 1), seed=85)
    both = cuda_lib.Context(pairs=[dict(fixed=f, moving=m, bins=64),
                                   dict(fixed=f16, moving=m16, bins=32, fixed_depth=12, moving_depth=12)], **kw)
    got, _, cnt = both.batch_eval(np.zeros(4, np.int32), prm, [1.0, 2.0], with_entropies=True)
    mi_o, h_o, cnt_o = oracle.mi_eval(f, m, 64, prm, [1.0, 2.0], nthreads=8)
    np.testing.assert_array_equal(cnt, cnt_o)
    assert np.all(np.abs(got - mi_o) <= 1e-6 * np.maximum(np.abs(mi_o), h_o[..., 2]) + 1e-12)
    for path in (cuda_lib.PATH_PLAIN, cuda_lib.PATH_BATCHED):
        H = ctx.hist(transforms=prm, path=path)
        for t in range(4):
            q16 = oracle.affine_q16(oracle.affine(prm[t], f.shape, (1, 1, 1), m.shape, (1, 1, 1)))
            np.testing.assert_array_equal(H[t], oracle.joint_hist(f, m, q16, 64)[0].astype(np.uint32))


@pytest.mark.parametrize("dtype,depth,offset", [(np.uint8, 8, 3), (np.uint8, 5, 0), (np.uint16, 12, 1), (np.uint16, 16, 5),
                                                (np.float32, 0, 1)])
def test_layouts_from_unaligned_device_volumes(cuda_lib, dtype, depth, offset):
    """Volumes used where they lie on the device: any element offset, voxel counts that leave a remainder of
    the eight-wide loads, values above the declared depth; then one context walks through its layouts (one
    pose, several, forced variants of every fetch) with the same histograms, also on another stream."""
    import torch

    rng = np.random.default_rng(86)
    shape, mshape = (7, 9, 13), (11, 6, 17)
    top = 2 if dtype == np.float32 else np.iinfo(dtype).max + 1
    f, m = ((rng.random(s).astype(dtype) if dtype == np.float32 else rng.integers(0, top, s, dtype=dtype)) for s in (shape, mshape))
    dev = []
    for a in (f, m):
        flat = torch.zeros(a.size + 16, dtype=getattr(torch, np.dtype(dtype).name), device="cuda")
        flat[offset:offset + a.size] = torch.from_numpy(a).reshape(-1).cuda()
        dev.append(flat[offset:offset + a.size].reshape(a.shape))
    kw = dict(bins=32, fixed_depth=depth or None, moving_depth=depth or None)
    ctx = cuda_lib.Context(dev[0], dev[1], **kw)
    for d in dev:
        d.zero_()  # the context has its own copy
    prm = phantoms.random_transforms(400, seed=87, t_mm=2, r_deg=15, s_range=(0.9, 1.1))
    mi_o, h_o, cnt_o = oracle.mi_eval(f, m, 32, prm, [1.0], fixed_depth=depth or None, moving_depth=depth or None, nthreads=8)
    ok = cnt_o > 0
    np.testing.assert_array_equal(ctx.fixed_bins(), oracle.bin_volume(f, 32, depth or None).reshape(shape))
    for n in (1, 5, 400):
        mi, _, cnt = ctx.eval(prm[:n], [1.0], with_entropies=True)
        np.testing.assert_array_equal(cnt, cnt_o[:n])
        g = ok[:n]
        assert np.all(np.abs(mi[g] - mi_o[:n][g]) <= 1e-6 * np.maximum(np.abs(mi_o[:n][g]), h_o[:n][g][..., 2]) + 1e-12)
    for v in (cuda_lib.HV_U32, cuda_lib.HV_U32_TEX, cuda_lib.HV_U32_QUAD) + ((cuda_lib.HV_U32_GATHER,) if 0 < depth <= 12 else ()):
        other = cuda_lib.Context(f, m, hist_variant=v, **kw)
        other.set_stream(torch.cuda.Stream())
        np.testing.assert_array_equal(other.hist(transforms=prm[:4]), ctx.hist(transforms=prm[:4]))

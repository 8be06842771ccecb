"""Device memory that calls take beyond the volumes."""
import numpy as np
import pytest

from paper_1909_10690_gb300 import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(autotune=False), dict(hist_variant=0, block_threads=1024)])
def test_only_the_chosen_variants_layout_without_timing(cuda_lib, kw):
    """A batched call that has nothing to time builds the one layout it reads: of 256^3 bytes the x-pairs take
    34 MB, every layout together 200."""
    import torch

    rng = np.random.default_rng(103)
    f, m = (rng.integers(0, 256, (256, 256, 256), dtype=np.uint8) for _ in range(2))
    ctx = cuda_lib.Context(f, m, bins=64, path="batched", **kw)
    prm = phantoms.random_transforms(4, seed=104, t_mm=3, r_deg=8, s_range=(0.95, 1.05))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx.eval(prm)
    taken = before - torch.cuda.mem_get_info()[0]
    assert ctx.selected_variant(4) == cuda_lib.HV_U32
    assert taken < 100e6, taken


def test_no_room_for_split_transforms(cuda_lib):
    """A batched call fails one allocation after another; where it is the split transforms' histograms, which it
    can do without, it keeps its transforms whole (one launch instead of two) with the same results."""
    f, m = phantoms.head_pair(shape=(64, 64, 64), spacing=(1, 1, 1), seed=105)
    kw = dict(bins=32, fixed_depth=12, moving_depth=12, autotune=False)
    prm = phantoms.random_transforms(160, seed=106, t_mm=3, r_deg=8, s_range=(0.95, 1.05))
    qs = [1.0, 1.5]
    want = cuda_lib.Context(f, m, path="plain", **kw).eval(prm, qs)
    lib = cuda_lib.load()
    launches = []
    try:
        for k in range(16):
            ctx = cuda_lib.Context(f, m, **kw)
            lib.mi_fault_alloc(k)
            try:
                got = ctx.eval(prm, qs)
            except cuda_lib.MIError as e:
                assert e.status == cuda_lib.MI_ENOMEM
                continue
            finally:
                lib.mi_fault_alloc(-1)
            np.testing.assert_allclose(got, want, rtol=1e-12, atol=1e-14)
            launches.append(ctx.last_kernel_ms()[1])
            for n in (160, 320):  # the context goes on, also with a larger call
                np.testing.assert_allclose(ctx.eval(prm[np.arange(n) % 160], qs)[:160], want, rtol=1e-12, atol=1e-14)
            if launches[-1] == 2:
                break  # no allocation failed
    finally:
        lib.mi_fault_alloc(-1)
    assert launches[-1] == 2 and 1 in launches[:-1], launches

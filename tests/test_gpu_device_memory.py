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

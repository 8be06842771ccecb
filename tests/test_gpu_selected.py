"""mi_selected_variant / mi_selected_config: the plain path answers for every transform count after any of its calls."""
import pytest

from paper_1909_10690_gb300 import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first,other", [(1, 10), (10, 1), (2, 3)])
def test_plain_choice_for_other_transform_counts(cuda_lib, first, other):
    f, m = phantoms.ellipsoid_pair(shape=(32, 32, 32), seed=107)
    prm = phantoms.random_transforms(10, seed=108, t_mm=3, r_deg=8)
    ctx = cuda_lib.Context(f, m, bins=32)
    assert ctx.selected_variant(other) == -1 and set(ctx.selected_config(first).values()) == {-1}
    ctx.eval(prm[:first])
    asked = ctx.selected_config(other)
    assert asked["variant"] == ctx.selected_variant(other) >= 0 and asked["ctas"] > 0
    ctx.eval(prm[:other])
    assert ctx.selected_config(other) == asked
    assert ctx.selected_variant(500) == -1  # the batched path has not been called

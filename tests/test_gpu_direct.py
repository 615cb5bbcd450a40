"""Small games in one launch (fsi_direct_kernel) against the tile path of the
same plan, bitwise: both evaluate the same integer.  The fused schedule always
takes the tiles, and so does a batch of many games (needs a GB300)."""
import numpy as np
import pytest

import paper_2601_01903_gb300 as fsi
from paper_2601_01903_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _values(B, d, seed, scale=1.0):
    return torch.as_tensor(scale * synthetic.Stream(seed, 3).normal(B << d).reshape(B, 1 << d), device="cuda")


@pytest.mark.parametrize("index", ["fsi", "sii", "bii", "stii", "ksii"])
@pytest.mark.parametrize("d,ell,B", [(2, 1, 3), (3, 2, 1), (4, 3, 2), (5, 4, 5), (6, 2, 1), (8, 2, 1), (9, 4, 3),
                                     (10, 3, 7), (11, 1, 2), (11, 4, 1)])
def test_direct_is_bitwise_the_tile_path(index, d, ell, B):
    v = _values(B, d, d * 10 + ell)
    plan = fsi.Plan(d, ell, "exact", max_batch=B, index=index)
    direct = plan.apply(v)
    plan.set_schedule(fused=True)
    assert torch.equal(direct, plan.apply(v))
    plan.check()


@pytest.mark.parametrize("scale", [0.0, 1e-310, 1e-290, 2.0 ** -990, 1e300])
def test_extreme_scales(scale):
    v = _values(2, 7, 4, scale)
    v[1, 5:] = 0.0
    plan = fsi.Plan(7, 3, "exact", max_batch=2)
    direct = plan.apply(v)
    plan.set_schedule(fused=True)
    assert torch.equal(direct, plan.apply(v))


def test_large_batch_takes_tiles_with_the_same_scores():
    # 176 scores x 2^10 values a game: 200 games are past the products of the rule
    v = _values(200, 10, 8)
    many = fsi.Plan(10, 3, "exact", max_batch=200).apply(v)
    few = fsi.Plan(10, 3, "exact", max_batch=1)
    for b in (0, 77, 199):
        assert torch.equal(few.apply(v[b:b + 1])[0], many[b])


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_value_is_reported(bad):
    v = _values(2, 6, 5)
    v[1, 3] = bad
    plan = fsi.Plan(6, 2, "exact", max_batch=2)
    good = plan.apply(v[:1])
    plan.check()
    assert torch.equal(plan.apply(v)[0], good[0])
    with pytest.raises(fsi.FsiError) as e:
        plan.check()
    assert e.value.status == 6

"""Few scores over many tiles: the combine's lanes per score (exact) and its
segments (float) against the fused schedule, bitwise, with tiles of equal and
of different exponents, and past the aligned exponent range (needs a GB300)."""
import pytest

import paper_2601_01903_gb300 as fsi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arith", ["exact", "f32", "f64"])
@pytest.mark.parametrize("d,ell,B", [(20, 3, 1), (20, 1, 3), (21, 2, 1), (22, 1, 3), (22, 2, 1), (23, 1, 1), (23, 3, 1),
                                     (24, 2, 1)])
@pytest.mark.parametrize("spread", [0, 12, 90])
def test_split_equals_fused(arith, d, ell, B, spread):
    dt = torch.float32 if arith == "f32" else torch.float64
    g = torch.Generator(device="cuda").manual_seed(d * 10 + ell)
    v = torch.rand(B, 1 << d, generator=g, device="cuda", dtype=dt) + 1.0  # one exponent
    if spread:  # every eighth tile smaller by 2^spread
        v.view(B, -1, 4096)[:, ::8] *= 2.0 ** -min(spread, 60 if arith == "f32" else spread)
    plan = fsi.Plan(d, ell, arith, max_batch=B)
    split = plan.apply(v)
    plan.set_schedule(fused=True, tiles_per_item=2)
    assert torch.equal(split, plan.apply(v))
    plan.check()

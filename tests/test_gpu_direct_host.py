"""Small games from host memory: read in place while few blocks read a game,
copied first beyond that; the device path's scores either way, bitwise (needs a
GB300)."""
import pytest

import paper_2601_01903_gb300 as fsi
from paper_2601_01903_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# bytes read by all blocks: 10 KB, 1.1 MB, just below and above 1.25 MB (10, 3: 176 KB
# a game), 1.9 MB; the last on the tile path (past the direct kernel's products)
@pytest.mark.parametrize("d,ell,B", [(8, 2, 1), (11, 4, 1), (10, 3, 7), (10, 3, 8), (11, 3, 4), (10, 3, 60)])
@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("zero_copy", [True, False])
def test_scores_of_host_games(d, ell, B, pinned, zero_copy):
    v = torch.as_tensor(synthetic.Stream(d, B).normal(B << d).reshape(B, 1 << d))
    plan = fsi.Plan(d, ell, "exact", max_batch=B)
    ref = plan.apply(v.cuda()).cpu()
    plan.set_host_zero_copy(zero_copy)
    host = v.pin_memory() if pinned else v
    for _ in range(2):
        assert torch.equal(plan.apply_host(host), ref)
    plan.check()

"""Batches on both sides of three tiles per SM, where the batch kernel changes
its register budget: bitwise the scores of one call per game (needs a GB300)."""
import numpy as np
import pytest

import paper_2601_01903_gb300 as fsi
from paper_2601_01903_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arith", ["exact", "f64", "f32"])
@pytest.mark.parametrize("top", [3, 4])
@pytest.mark.parametrize("ds", [[6], [12, 13, 8, 10], [18] * 7 + [15], [18] * 7 + [15, 12], [19, 19, 19, 17, 9]])
def test_batch_matches_calls_per_game(arith, top, ds):
    # (456 tiles of 4096 values are three for each of 152 SMs)
    games, vo, po = [], 0, 0
    for k, d in enumerate(ds):
        ell = 1 + (k + top - 1) % top
        games.append((d, ell, vo, po))
        vo += 1 << d
        po += synthetic.n_scores(d, ell)
    g = torch.Generator(device="cuda").manual_seed(len(ds))
    v = torch.randn(vo, generator=g, device="cuda", dtype=torch.float32 if arith == "f32" else torch.float64)
    batch = fsi.Batch(games, arith)
    phi = torch.full((po,), float("nan"), device="cuda", dtype=v.dtype)
    ref = torch.zeros_like(phi)
    batch.apply_per_game(v, ref)
    for schedule in ((1, 64), (3, 16)):
        batch.set_schedule(*schedule)
        for _ in range(2):
            batch.apply(v, phi.fill_(float("nan")))
            batch.check()
            if arith == "exact":
                assert torch.equal(phi, ref)
            else:
                unit = 2.0 ** -24 if arith == "f32" else 2.0 ** -53
                bound = 512 * unit * float(v.abs().max()) * 2.0 ** (max(ds) / 2)
                assert float((phi - ref).abs().max()) <= bound

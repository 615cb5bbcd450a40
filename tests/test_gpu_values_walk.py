"""Blocks of the split-digit value function (masked_game_split.cu) that walk
several tiles: the row sums of a tile are read by one warp of a row group
while the others are on their way to the next tile, so the same call many
times has to give the same bits, and the oracle's values (needs a GB300).

Tolerances as in test_gpu_values_split.py: 300 roundings of a few times max|v|."""
import numpy as np
import pytest

import paper_2601_01903_gb300 as fsi
from paper_2601_01903_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {torch.float64: 1.3e-13, torch.float32: 7e-5}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("d,h1,h2,B,n_bg,slow", [
    (15, 40, 20, 1, 1, False), (15, 64, 64, 1, 1, False), (13, 40, 20, 3, 1, False), (9, 32, 40, 60, 1, False),
    (13, 40, 70, 2, 3, False), (13, 100, 24, 3, 1, False), (11, 24, 30, 20, 1, True), (12, 40, 24, 6, 2, True)])
def test_repeated_calls_agree(oracle_mod, dtype, d, h1, h2, B, n_bg, slow):
    m = synthetic.random_mlp(d, h1, h2, d + h1)
    m.b1, m.b2 = 0.1 * synthetic.Stream(d, 5).normal(h1), 0.1 * synthetic.Stream(d, 6).normal(h2)
    x = synthetic.gaussian_instances(B, d, h2)
    if slow:
        x[::2, 3] = 1e9  # every other instance leaves the fixed-point range
    rows = np.zeros((1, d)) if n_bg == 1 else synthetic.gaussian_instances(n_bg, d, 3)
    dm, dx, dr = fsi.DeviceMLP(m), torch.as_tensor(x, device="cuda"), torch.as_tensor(rows, device="cuda")
    calls = [fsi.masked_game_interventional(dm, dx, dr, dtype=dtype) for _ in range(24)]
    assert all(torch.equal(calls[0], c) for c in calls[1:])
    got = calls[0].cpu().numpy().astype(np.float64)
    for b in sorted({0, B // 2, B - 1}):
        ref = oracle_mod.masked_game_interventional(m, x[b], rows)
        assert np.max(np.abs(got[b] - ref)) <= TOL[dtype] * np.max(np.abs(ref))

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
    (13, 40, 70, 2, 3, False), (13, 100, 24, 3, 1, False),
    (9, 40, 70, 60, 1, False), (9, 100, 128, 50, 1, False), (8, 70, 100, 90, 2, True), (11, 24, 30, 20, 1, True), (12, 40, 24, 6, 2, True)])
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


def _sensitivity(m, x, rows):
    """What a relative change of 1 in every operand can move a value by (first
    order), [instance, coalition]."""
    t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64))
    cdf = lambda z: 0.5 * (1 + torch.erf(z / 2 ** 0.5))
    slope = lambda z: (cdf(z) + z * torch.exp(-z * z / 2) / 6.283185307179586 ** 0.5).abs()
    d = x.shape[1]
    on = ((np.arange(1 << d)[:, None] >> np.arange(d)) & 1).astype(bool)
    out = []
    for v in x:
        z = t(np.where(on, v, rows))
        z1 = z @ t(m.W1).T + t(m.b1)
        a1 = z1 * cdf(z1)
        z2 = a1 @ t(m.W2).T + t(m.b2)
        s1 = a1.abs() + slope(z1) * (z.abs() @ t(m.W1).abs().T + t(m.b1).abs())
        s2 = (z2 * cdf(z2)).abs() + slope(z2) * (s1 @ t(m.W2).abs().T + t(m.b2).abs())
        out.append(s2 @ t(m.W3).reshape(-1).abs() + abs(float(m.b3[0])))
    return torch.stack(out)


@pytest.mark.parametrize("dtype,scale", [(torch.float64, 300.0), (torch.float32, 1e12)])
@pytest.mark.parametrize("h1,h2", [(40, 48), (100, 40), (96, 128)])
def test_some_rows_of_many_tiles_outside_the_range(dtype, scale, h1, h2):
    """Two large features: the coalitions without them leave the fixed point, the
    others of the same tiles do not; blocks walk on to the next tiles."""
    d, B = 9, 50
    m = synthetic.random_mlp(d, h1, h2, 3)
    m.b3[:] = 0.05
    x = synthetic.gaussian_instances(B, d, 8)
    x[:, [2, 8]] *= scale
    x[::7] = synthetic.gaussian_instances(len(x[::7]), d, 9)  # and ordinary instances between
    wide = synthetic.MLP(np.vstack([m.W1, np.zeros((129 - h1, d))]), np.zeros(129),
                         np.hstack([m.W2, np.zeros((h2, 129 - h1))]), m.b2, m.W3, m.b3)
    got = [fsi.masked_game(m, x, np.zeros(d), dtype=dtype) for _ in range(8)]
    assert all(torch.equal(got[0], g) for g in got[1:])
    yard = fsi.masked_game(wide, x, np.zeros(d), dtype=dtype)  # masked_game_kernel
    unit = 2.0 ** -53 if dtype == torch.float64 else 2.0 ** -24
    assert bool(((got[0].double() - yard.double()).abs().cpu() <= 16 * unit * _sensitivity(m, x, np.zeros(d))).all())

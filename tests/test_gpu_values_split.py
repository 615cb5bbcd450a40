"""The value function's split-digit tensor-core path (masked_game_split.cu)
against the oracle at the edges of its tiles: widths around the K and N
granules, the smallest d, several background rows, scales that leave the
fixed-point range, non-finite features (needs a GB300).

Tolerances.  float64: both sides round every dot product of at most d + h1 +
h2 < 300 terms, each by 2^-53 of values below a few times max|v|: 300 * 4 *
1.1e-16 = 1.3e-13.  float32: the same with 2^-24: 300 * 4 * 6e-8 = 7e-5."""
import numpy as np
import pytest

import paper_2601_01903_gb300 as fsi
from paper_2601_01903_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {torch.float64: 1.3e-13, torch.float32: 7e-5}


def _model(d, h1, h2, seed):
    m = synthetic.random_mlp(d, h1, h2, seed)
    st = synthetic.Stream(seed, 5)
    m.b1, m.b2, m.b3 = 0.1 * st.normal(h1), 0.1 * st.normal(h2), 0.1 * st.normal(1)
    return m


def _check(oracle_mod, m, x, rows, dtype):
    rows = np.atleast_2d(rows)
    if len(rows) == 1:
        got = fsi.masked_game(m, x, rows[0], dtype=dtype)
    else:
        got = fsi.masked_game_interventional(m, x, rows, dtype=dtype)
    got = got.cpu().numpy().astype(np.float64)
    for b in range(len(x)):
        ref = oracle_mod.masked_game_interventional(m, x[b], rows)
        assert np.max(np.abs(got[b] - ref)) <= TOL[dtype] * np.max(np.abs(ref))


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("d,h1,h2,B,n_bg", [
    (7, 1, 1, 3, 1), (7, 24, 24, 1, 1), (8, 16, 33, 2, 1), (8, 17, 64, 1, 2), (9, 32, 65, 2, 1), (8, 33, 31, 2, 3),
    (10, 63, 128, 1, 1), (9, 64, 16, 3, 1), (8, 65, 17, 2, 2), (9, 127, 96, 1, 1), (10, 128, 127, 2, 1),
    (8, 129, 40, 1, 2), (15, 40, 20, 1, 1)])
def test_widths_and_rows(oracle_mod, dtype, d, h1, h2, B, n_bg):
    x = synthetic.gaussian_instances(B, d, d + h1)
    rows = np.zeros((1, d)) if n_bg == 1 else synthetic.gaussian_instances(n_bg, d, 3)
    _check(oracle_mod, _model(d, h1, h2, h2), x, rows, dtype)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("scale", [1e-30, 1e-4, 0.2, 30.0, 1e5, 1e9])
def test_scales(oracle_mod, dtype, scale):
    m = _model(8, 40, 50, 1)
    m.b1[:] = 0.0
    x = synthetic.gaussian_instances(3, 8, 2) * scale
    x[1] *= 1e-3  # instances of different scales in one call
    _check(oracle_mod, m, x, np.zeros(8), dtype)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("what", ["lone_feature", "zero_W2", "zero_W3", "zero_x", "large_W2"])
def test_degenerate_models(oracle_mod, dtype, what):
    m = _model(9, 36, 70, 4)
    x = synthetic.gaussian_instances(2, 9, 5)
    if what == "lone_feature":
        x[0, 3] = 1e4
        x[1, 8] = -1e7
    elif what == "zero_x":
        x[:] = 0.0
    elif what == "large_W2":
        m.W2 = m.W2 * 1e4
    else:
        setattr(m, what[5:], np.zeros_like(getattr(m, what[5:])))
    _check(oracle_mod, m, x, np.zeros(9), dtype)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("feature", [2, 8])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_feature_stays_in_its_coalitions(oracle_mod, dtype, feature, bad):
    m = _model(9, 48, 40, 6)
    x = synthetic.gaussian_instances(2, 9, 7)
    ref = np.stack([oracle_mod.masked_game(m, r, np.zeros(9)) for r in x])
    x[1, feature] = bad
    got = fsi.masked_game(m, x, np.zeros(9), dtype=dtype).cpu().numpy().astype(np.float64)
    has = (np.arange(512) >> feature & 1).astype(bool)
    assert np.max(np.abs(got[0] - ref[0])) <= TOL[dtype] * np.abs(ref).max()
    assert np.max(np.abs(got[1][~has] - ref[1][~has])) <= TOL[dtype] * np.abs(ref).max()
    assert not np.isfinite(got[1][has]).any()

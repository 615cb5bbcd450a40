"""The tensor-core value function at the edges of its launch shapes: listed
rows per instance around the staging rule, features around the shared-memory
rows of W1, few tiles with many background rows (clusters), a non-finite
feature (needs a GB300).  Bound: TC_EMU_TOL of test_gpu_masked_game.py, the
BF16 emulation's."""
import numpy as np
import pytest

import paper_2601_01903_gb300 as fsi
from paper_2601_01903_gb300 import synthetic
from test_gpu_masked_game import TC_EMU_TOL, _forward_bf16, _inputs, _rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _model(d, seed):
    m = synthetic.random_mlp(d, 128, 128, seed)
    st = synthetic.Stream(seed, 5)
    m.b1, m.b2, m.b3 = 0.1 * st.normal(128), 0.1 * st.normal(128), 0.1 * st.normal(1)
    return m


def _rows(n, d, seed):
    return 0.5 * synthetic.gaussian_instances(n, d, seed)


def _emulated(m, x, rows, masks, d):
    return np.mean([_forward_bf16(m, _inputs(x, r, masks, d)) for r in rows], axis=0)


@pytest.mark.parametrize("d,B,K,n_bg", [(1, 3, 2, 1), (5, 200, 1, 1), (16, 9, 31, 2), (16, 9, 32, 1), (17, 7, 33, 1),
                                        (9, 2, 127, 3), (32, 2, 130, 9), (12, 1, 1, 40)])
def test_listed_rows(d, B, K, n_bg):
    m, x, rows = _model(d, d), synthetic.gaussian_instances(B, d, 7), _rows(n_bg, d, 3)
    coal = synthetic.Stream(K, 2).integers(0, (1 << d) - 1, B * K).astype(np.uint32).reshape(B, K)
    got = fsi.masked_game_tc(m, x, rows, coalitions=coal).cpu().numpy().astype(np.float64)
    for b in range(B):
        ref = _emulated(m, x[b], rows, coal[b].astype(np.int64), d)
        assert np.max(np.abs(got[b] - ref)) <= TC_EMU_TOL * max(np.abs(ref).max(), 0.1)


@pytest.mark.parametrize("d,B,n_bg", [(7, 1, 1), (7, 1, 50), (8, 3, 2), (10, 2, 7), (15, 1, 2), (17, 2, 1), (18, 1, 3),
                                      (11, 40, 5)])
def test_dense_tiles_and_clusters(d, B, n_bg):
    m, x, rows = _model(d, d + 1), synthetic.gaussian_instances(B, d, 8), _rows(n_bg, d, 4)
    got = fsi.masked_game_tc(m, x, rows).cpu().numpy().astype(np.float64)
    again = fsi.masked_game_tc(m, x, rows).cpu().numpy().astype(np.float64)
    assert np.array_equal(got, again)
    masks = np.arange(1 << d, dtype=np.int64) if d <= 12 else synthetic.Stream(d, 1).integers(0, (1 << d) - 1, 2000)
    for b in range(0, B, max(1, B // 3)):
        assert _rel(got[b][masks], _emulated(m, x[b], rows, masks, d)) <= TC_EMU_TOL


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_feature(bad):
    d = 9
    m, x = _model(d, 2), synthetic.gaussian_instances(2, d, 9)
    clean = fsi.masked_game_tc(m, x, np.zeros(d)).cpu().numpy()
    x[1, 8] = bad
    got = fsi.masked_game_tc(m, x, np.zeros(d)).cpu().numpy()
    has = np.arange(1 << d) >> 8 & 1 == 1
    assert np.array_equal(got[0], clean[0]) and np.array_equal(got[1][~has], clean[1][~has])
    assert not np.isfinite(got[1][has]).any()

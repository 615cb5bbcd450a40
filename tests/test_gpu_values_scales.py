"""The split-digit value function (masked_game_split.cu) on models whose units
have different scales and instances whose features do, coalition by coalition
(needs a GB300).

The same model with its first layer padded to 129 hidden units by units
without weights takes masked_game_kernel, which rounds every operation at its
own scale: it is the yardstick.  Errors are taken against a forward pass in
extended precision and divided by what a relative change of 1 in every
operand of that coalition can move its value by (first order), so that one
number serves coalitions of every size.  Both sides round operands at 2^-53
(float64) or 2^-24 (float32); they sum in different orders and with different
GELUs, so the largest and the mean error of the split-digit path may be up to
twice the yardstick's."""
import numpy as np
import pytest

import paper_2601_01903_gb300 as fsi
from paper_2601_01903_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L = np.longdouble


def _cdf(z):
    """The normal distribution function by erf's series of positive terms,
    erf(x) = 2 / sqrt(pi) exp(-x^2) sum 2^n x^(2n+1) / (2n+1)!!  (beyond 9, 0 or 1)."""
    x = np.minimum(np.abs(z), L(9)) / np.sqrt(L(2))
    pi = L("3.14159265358979323846264338327950288")
    s = t = x.copy()
    for n in range(1, 400):
        t = t * (2 * x * x / L(2 * n + 1))
        s = s + t
        if not np.any(t > s * L(1e-24)):
            break
    erf = np.where(np.abs(z) > 9, L(1), 2 / np.sqrt(pi) * np.exp(-x * x) * s)
    return (1 + np.sign(z) * erf) / 2


def _forward(m, x, base):
    """Values of every coalition of one instance, and their sensitivity."""
    d = len(x)
    on = ((np.arange(1 << d)[:, None] >> np.arange(d)) & 1).astype(bool)
    z = np.where(on, x, base).astype(L)
    W1, b1, W2, b2, W3 = (np.asarray(a, dtype=np.float64).astype(L) for a in (m.W1, m.b1, m.W2, m.b2, m.W3))
    W3, b3 = W3.reshape(-1), L(float(np.asarray(m.b3).reshape(-1)[0]))
    slope = lambda y: np.abs(_cdf(y) + y * np.exp(-y * y / 2) / np.sqrt(L(6.283185307179586)))
    z1 = z @ W1.T + b1
    a1 = z1 * _cdf(z1)
    z2 = a1 @ W2.T + b2
    a2 = z2 * _cdf(z2)
    f = a2 @ W3 + b3
    s1 = np.abs(a1) + slope(z1) * (np.abs(z) @ np.abs(W1).T + np.abs(b1))
    s2 = np.abs(a2) + slope(z2) * (s1 @ np.abs(W2).T + np.abs(b2))
    return f, s2 @ np.abs(W3) + abs(b3)


def _padded(m):
    n = 129 - len(m.b1)
    return synthetic.MLP(np.vstack([m.W1, np.zeros((n, m.W1.shape[1]))]), np.concatenate([m.b1, np.zeros(n)]),
                         np.hstack([m.W2, np.zeros((len(m.b2), n))]), m.b2, m.W3, m.b3)


def _values(m, x, rows, dtype):
    if len(rows) == 1:
        return fsi.masked_game(m, x, rows[0], dtype=dtype).cpu().numpy()
    return fsi.masked_game_interventional(m, x, rows, dtype=dtype).cpu().numpy()


def _errors(m, x, rows, dtype):
    """Scaled errors [instance, coalition] of the path and of the yardstick."""
    got, yard = _values(m, x, rows, dtype), _values(_padded(m), x, rows, dtype)
    e = np.empty((2,) + got.shape)
    for b in range(len(x)):
        fs = [_forward(m, x[b], r) for r in rows]
        f, s = sum(f for f, _ in fs) / len(rows), sum(s for _, s in fs) / len(rows)
        s = np.maximum(s, L(1e-300))
        e[0, b], e[1, b] = np.abs(got[b].astype(L) - f) / s, np.abs(yard[b].astype(L) - f) / s
    return e


def _check(m, x, rows):
    for dtype in (torch.float64, torch.float32):
        e, y = _errors(m, x, np.atleast_2d(rows), dtype)
        assert np.all(np.isfinite(e))
        assert e.max() <= 2 * y.max(), (dtype, e.max(), y.max())
        assert e.mean() <= 2 * y.mean(), (dtype, e.mean(), y.mean())


def _model(d, h1, h2, seed, bias=0.1):
    m = synthetic.random_mlp(d, h1, h2, seed)
    st = synthetic.Stream(seed, 5)
    m.b1, m.b2, m.b3 = bias * st.normal(h1), bias * st.normal(h2), bias * st.normal(1)
    return m


def _scaled(m, what, k):
    c = 2.0 ** k
    if what == "unit1":  # one unit of layer 1, undone in layer 2
        m.W1[0] *= c
        m.b1[0] *= c
        m.W2[:, 0] /= c
    else:  # one unit of layer 2, undone in layer 3
        m.W2[0] *= c
        m.b2[0] *= c
        m.W3[0, 0] /= c
    return m


@pytest.mark.parametrize("what", ["unit1", "unit2"])
@pytest.mark.parametrize("k", [-28, -20, -14, -10, -7, -5, -3, 0, 3, 5, 7, 10, 14, 20, 28])
def test_one_unit_of_another_scale(what, k):
    x = synthetic.gaussian_instances(1, 8, 11)
    _check(_scaled(_model(8, 40, 48, 2), what, k), x, np.zeros(8))


@pytest.mark.parametrize("k", [-9, -6, 6, 9, 24])
def test_half_of_the_units_of_another_scale(k):
    m, c = _model(8, 66, 30, 3), 2.0 ** k
    m.W1[::2] *= c
    m.b1[::2] *= c
    m.W2[:, ::2] /= c
    _check(m, synthetic.gaussian_instances(1, 8, 12), np.zeros(8))
    m, c = _model(8, 30, 66, 3), 2.0 ** k
    m.W2[::2] *= c
    m.b2[::2] *= c
    m.W3[:, ::2] /= c
    _check(m, synthetic.gaussian_instances(1, 8, 12), np.zeros(8))


@pytest.mark.parametrize("b", [-20.0, -40.0, -1e3, -6e4, -1e8, 1e3])
@pytest.mark.parametrize("layer,others", [(1, 0.1), (2, 0.1), (1, 0.0)])
def test_outlying_bias(layer, b, others):
    m = _model(8, 40, 48, 4, others)
    (m.b1 if layer == 1 else m.b2)[3] = b
    _check(m, synthetic.gaussian_instances(1, 8, 13), np.zeros(8))


@pytest.mark.parametrize("h1,h2", [(12, 20), (40, 48), (128, 96)])
@pytest.mark.parametrize("k", [2, 4, 5, 8])
def test_unit_that_outweighs_the_others_where_it_is_active(h1, h2, k):
    m = _model(8, h1, h2, 4)
    m.W2[:, 3] *= 2.0 ** k
    m.b1[3] = -5.0
    _check(m, synthetic.gaussian_instances(2, 8, 13), np.zeros(8))
    m = _model(8, h1, h2, 4)
    m.W3[0, 3] *= 2.0 ** k
    m.b2[3] = -4.0
    _check(m, synthetic.gaussian_instances(1, 8, 13), np.zeros(8))


@pytest.mark.parametrize("bias", [0.1, 0.0])
@pytest.mark.parametrize("scale", [30.0, 1e3, 1e4, 1e5, 1e12])
def test_two_large_features(scale, bias):
    m, x = _model(9, 36, 40, 5, bias), synthetic.gaussian_instances(1, 9, 14)
    x[0, [2, 8]] *= scale
    _check(m, x, np.zeros(9))


@pytest.mark.parametrize("scale", [1e-5, 1e-2, 0.1, 1.0, 20.0])
def test_coalitions_of_small_values(scale):
    """No biases: the small coalitions have values of the size of their features."""
    x = synthetic.gaussian_instances(2, 8, 15)
    x[0, ::2] *= 0.01
    _check(_model(8, 48, 64, 6, 0.0), x * scale, np.zeros(8))


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("h1,h2", [(16, 20), (64, 64), (100, 128)])
def test_features_of_zero_without_biases_give_b3(dtype, h1, h2):
    """GELU(0) is 0 in every layer."""
    m, x = _model(8, h1, h2, 6, 0.0), synthetic.gaussian_instances(3, 8, 15)
    x[1, :4] = 0.0
    x[2] = 0.0
    for b3 in (0.0, 0.3):
        m.b3[:] = b3
        v = fsi.masked_game(m, x, np.zeros(8), dtype=dtype)
        exact = torch.tensor(b3, dtype=dtype, device="cuda")
        assert bool((v[:, 0] == exact).all() and (v[1, :16] == exact).all() and (v[2] == exact).all())


def test_background_rows_of_different_scales():
    rows = synthetic.gaussian_instances(3, 8, 16) * np.array([[1e-3], [1.0], [50.0]])
    _check(_model(8, 64, 32, 7), synthetic.gaussian_instances(2, 8, 17), rows)


@pytest.mark.parametrize("h1,h2", [(1, 4), (2, 2), (4, 3), (16, 128), (128, 128)])
def test_widths(h1, h2):
    _check(_model(8, h1, h2, 8), synthetic.gaussian_instances(1, 8, 18), np.zeros(8))


def test_few_tiles_share_two_blocks_each():
    """At most half as many tiles as SMs: two blocks a tile, both on either route."""
    m, x = _model(7, 40, 48, 9), synthetic.gaussian_instances(3, 7, 19)
    x[1, 2] = 1e9
    _check(m, x, np.zeros(7))

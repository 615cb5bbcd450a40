"""The student's step over the edges of its tiles: batches, widths and output
counts below, at and just past the 128 x 128 tiles, the 64-wide K blocks and
the K slices, alternating batch sizes on one handle, against the oracle."""
import numpy as np
import pytest

from oracle import student as so
from paper_2601_01903_gb300 import student as st

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# Four BF16 roundings to the neighbouring value, relative to the
# root-sum-square scale of an entry (see test_gpu_student.py).
FLIP = 4 * 2.0 ** -8


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _batch(d, n_out, B, seed):
    rng = np.random.default_rng(seed)
    labels = (rng.normal(size=(B, n_out)) * 0.1).astype(np.float32)
    labels[:, 0] = 0.2
    return rng.normal(size=(B, d)).astype(np.float32), labels, rng.normal(size=B).astype(np.float32)


@pytest.mark.parametrize("d,H,n_out,batches", [
    (8, 8, 2, (1, 33)),
    (8, 40, 37, (127, 64, 129)),
    (16, 136, 137, (300, 257)),
    (24, 200, 301, (513,)),
    (72, 64, 73, (96,)),
    (16, 520, 16, (1100, 31)),
])
def test_gradients_and_scores_at_tile_edges(d, H, n_out, batches):
    params = st.init_params(d, H, n_out, 7, out_scale=0.3)
    p64 = params.astype(np.float64)
    s = st.Student(d, H, n_out, max(batches), params)
    sizes = (H * d, H, H * H, H, n_out * H, n_out)
    for B in batches + batches[:1]:
        x, labels, target = _batch(d, n_out, B, B)
        loss = s.gradients(_dev(x), _dev(labels), _dev(target), 0.2)
        s.check()
        g = s.grads().astype(np.float64)
        ref_loss, ref = so.loss_and_grads(p64, x, labels, target, 0.2, d, H, n_out, emulate_bf16=True)
        mag = so.grad_magnitudes(p64, x, labels, target, 0.2, d, H, n_out)
        assert abs(loss.item() - ref_loss) <= 1e-4 * abs(ref_loss)
        o = 0
        for name, n in zip(("W1", "b1", "W2", "b2", "W3", "b3"), sizes):
            bad = np.abs(g[o:o + n] - ref[o:o + n]) > FLIP * mag[o:o + n] + 1e-30
            assert not bad.any(), (B, name, int(bad.sum()))
            o += n
        phi = s.predict(_dev(x), _dev(target), 0.2).cpu().numpy().astype(np.float64)
        f = so.forward(p64, x, d, H, n_out, emulate_bf16=True)
        want = so.project(f["Y"], target, 0.2)
        m = so.output_magnitudes(p64, x, d, H, n_out)
        m[:, 1:] += m[:, 1:].mean(axis=1, keepdims=True)
        assert np.all(phi[:, 0] == np.float32(0.2))
        assert np.all(np.abs(phi[:, 1:] - want[:, 1:]) <= FLIP * m[:, 1:] + 1e-6 * np.abs(target)[:, None])

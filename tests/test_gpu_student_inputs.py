"""Inputs of the explainer's residual check in the forms that callers hand them
in (needs a GB300)."""
import numpy as np
import pytest

from paper_2601_01903_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _explainer():
    from paper_2601_01903_gb300 import student
    return student.Explainer(synthetic.random_mlp(8, 128, 128, 3), 2, hidden=128, batch=64, seed=5)


def test_residuals_take_any_baseline_tensor():
    ex = _explainer()
    x = torch.as_tensor(synthetic.gaussian_instances(150, 8, 4), dtype=torch.float32, device="cuda")
    phi = ex.predict_raw(x, ex.targets(x.double()))
    base = synthetic.Stream(6, 7).integers(-3, 3, 8) * 0.125  # exact in float32
    ex.baseline = torch.as_tensor(base, dtype=torch.float64, device="cuda")
    ref = ex.residuals(x, phi)
    strided = torch.as_tensor(np.stack([base, base], axis=1), device="cuda")[:, 0]
    for form in (torch.as_tensor(base, dtype=torch.float32, device="cuda"), torch.as_tensor(base), strided, base):
        ex.baseline = form
        assert torch.equal(ex.residuals(x, phi), ref)
    assert torch.equal(ex.residuals(x.cpu(), phi), ref)


@pytest.mark.parametrize("shape", [(7,), (9,), (2, 7)])
def test_residuals_refuse_a_baseline_of_another_width(shape):
    ex = _explainer()
    x = torch.zeros(5, 8, device="cuda")
    phi = ex.predict_raw(x, ex.targets(x.double()))
    ex.baseline = torch.zeros(shape, dtype=torch.float64, device="cuda")
    with pytest.raises(ValueError):
        ex.residuals(x, phi)

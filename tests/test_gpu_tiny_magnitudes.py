"""FP32 magnitudes near and below the smallest normal number, one object by the whole-grid transform."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-30, 1e-38, 1e-40, 1e-41])
def test_powers_do_not_depend_on_the_unit(scale):
    """Tolerance as in test_gpu_transform (1.2e-5), against the FP64 path on the same FP32 magnitudes."""
    import torch
    from paper_2105_04006_gb300 import build
    build.build()
    import paper_2105_04006_gb300 as lsp
    r = np.random.default_rng(3)
    t = np.sort(60000 + r.uniform(0, 400, 12_000))
    y = np.sin(2 * np.pi * 1.37 * t) + 0.5 * r.normal(size=t.size)
    g = lsp.Grid(1.3, 1.44, 10_007)
    t, y = torch.tensor(t, device="cuda"), torch.tensor((y * scale).astype(np.float32), device="cuda")
    p, _ = lsp.periodogram(t, y, g)
    ref, _ = lsp.periodogram(t, y.double(), g, precision="fp64")
    assert 0.5 < float(ref.max()) <= 1.0  # amplitude 1 in noise of 0.5: two thirds of the variance
    assert float((p.double() - ref).abs().max()) <= 1.2e-5

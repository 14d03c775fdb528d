"""FP32 sums of many observations in few cells of the transform's grid, where
the rounding of the fixed-point cells, not the window, sets the error.

Reference: the FP64 pairwise kernels on the same FP32 inputs.  Tolerances: the
standard periodogram 1.2e-5 (see test_gpu_transform: the window, the FP32
transform, and a denominator that magnifies them by up to 10; the cells' own
rounding adds about 2.4 sqrt(N) 2^-30 of the sum of the weights, 2e-6 at 1e6
observations), the generalized one the library's 1e-4.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    from paper_2105_04006_gb300 import build
    build.build()
    import paper_2105_04006_gb300 as lsp
    return lsp, torch, torch.device("cuda", 0)


def _batch(env, counts, days, sigma, seed):
    lsp, torch, dev = env
    r = np.random.default_rng(seed)
    t = [np.sort(60000 + r.uniform(0, days, n)) for n in counts]
    dy = [0.1 * np.exp(sigma * r.normal(size=n)) for n in counts]
    y = [0.4 * np.sin(2 * np.pi * 1.37 * a) + e * r.normal(size=a.size) + 3.0 for a, e in zip(t, dy)]
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    n_f = 700
    g = lsp.Grid(1.3, 1.3 + n_f * 1.176e-4, n_f)
    t, y, dy = np.concatenate(t), np.concatenate(y).astype(np.float32), np.concatenate(dy).astype(np.float32)
    return [torch.tensor(a, device=dev) for a in (t, y, dy, off)] + [g]


@pytest.mark.parametrize("counts,days", [([1_000_000, 300], 27.0), ([4095, 4096, 4097], 27.0), ([4095, 4096, 4097], 1.5),
                                         ([70_000, 4099], 4000.0)])
def test_standard(env, counts, days):
    lsp, torch, _ = env
    t, y, _, off, g = _batch(env, counts, days, 0.0, 41)
    p, _ = lsp.batch(t, y, off, g, return_power=True)
    ref, _ = lsp.batch(t, y.double(), off, g, return_power=True, precision="fp64", k_reseed=16)
    assert float((p.double() - ref).abs().max()) <= 1.2e-5


@pytest.mark.parametrize("counts,days", [([3_000_000, 300], 27.0), ([4095, 4096, 4097], 27.0)])
def test_generalized(env, counts, days):
    lsp, torch, _ = env
    t, y, dy, off, g = _batch(env, counts, days, 1.5, 43)
    p, _ = lsp.batch_gls(t, y, dy, off, g, return_power=True)
    ref, _ = lsp.batch_gls(t, y.double(), dy.double(), off, g, return_power=True, precision="fp64")
    assert float((p.double() - ref).abs().max()) <= 1e-4


def test_repeats_are_bit_identical(env):
    lsp, torch, _ = env
    t, y, dy, off, g = _batch(env, [9000, 5000], 27.0, 1.5, 47)
    a, _ = lsp.batch_gls(t, y, dy, off, g, return_power=True)
    b, _ = lsp.batch_gls(t, y, dy, off, g, return_power=True)
    assert torch.equal(a, b)

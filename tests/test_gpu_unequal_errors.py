"""Generalized periodogram (FP32) of light curves whose error bars differ
widely: the weights 1/dy^2 span up to 1e5, and many of them share few cells of
the transform's grid.

Reference: the FP64 generalized periodogram on the same FP32 inputs.  Tolerance:
the library's 1e-4 in the normalised power, as in test_gpu_gls.  (An FP32
emulation of the kernel with scales from the sums of the weights stays below
4e-6 on these shapes, the pairwise kernel's FP32 sums below 9e-5, and scales
from counts times the largest weight reach 5e-2.)
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 1e-4
COUNTS = [41, 300, 2000, 5000, 20_000]


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    from paper_2105_04006_gb300 import build
    build.build()
    import paper_2105_04006_gb300 as lsp
    return lsp, torch, torch.device("cuda", 0)


def _times(cadence, n, r):
    if cadence == "night":
        t = 60000.3 + r.uniform(0, 0.1, n)
    elif cadence == "month":
        t = 60000 + r.uniform(0, 27, n)
    elif cadence == "seasons":
        t = 60000 + 365.25 * r.integers(0, 10, n) + r.uniform(0, 150, n)
    else:  # most of them in ten nights
        k = int(0.8 * n)
        t = np.concatenate([60000.3 + r.integers(0, 10, k) + r.uniform(0, 0.3, k), 60000 + r.uniform(0, 3650, n - k)])
    return np.sort(t)


def _errors(kind, n, r):
    if kind == "lognormal":
        return 0.1 * np.exp(1.5 * r.normal(size=n))
    dy = np.full(n, 0.1)
    if kind == "few":  # one in a hundred 30 times smaller
        dy[r.choice(n, max(1, n // 100), replace=False)] /= 30
    else:  # one alone
        dy[r.integers(n)] /= kind
    return dy


def _light_curve(cadence, kind, n, seed):
    r = np.random.default_rng(seed + n)
    t, dy = _times(cadence, n, r), _errors(kind, n, r)
    y = 0.4 * np.sin(2 * np.pi * 1.37 * t) + dy * r.normal(size=n) + 3.0
    return t, y.astype(np.float32), dy.astype(np.float32)


@pytest.mark.parametrize("cadence", ["night", "month", "seasons", "ten_nights"])
@pytest.mark.parametrize("kind", [30, 100, 300, "few", "lognormal"])
def test_batch_of_unequal_errors(env, cadence, kind):
    lsp, torch, dev = env
    segs = [_light_curve(cadence, kind, n, 17) for n in COUNTS]
    t, y, dy = (np.concatenate([s[i] for s in segs]) for i in range(3))
    off = torch.tensor(np.concatenate([[0], np.cumsum(COUNTS)]).astype(np.int64), device=dev)
    n_f = 4111
    g = lsp.Grid(1.2, 1.2 + n_f * 1.176e-4, n_f)
    td, yd, ed = (torch.tensor(a, device=dev) for a in (t, y, dy))
    p, pk = lsp.batch_gls(td, yd, ed, off, g, return_power=True)
    ref, _ = lsp.batch_gls(td, yd.double(), ed.double(), off, g, return_power=True, precision="fp64")
    err = (p.double() - ref).abs().amax(dim=1).cpu().numpy()
    if cadence == "night":
        # a fraction of a cycle of data: near singular on every bin, which either FP32 path re-evaluates in FP64
        # from FP32 magnitudes that do not fix the power to 1e-4; the two have to agree
        q, _ = lsp.batch_gls(td, yd, ed, off, g, return_power=True, k_reseed=8)
        err = (p - q).abs().amax(dim=1).cpu().numpy()
    assert err.max() <= TOL, dict(zip(COUNTS, err))
    np.testing.assert_array_equal(lsp.peaks_to_numpy(pk)["idx"], p.argmax(dim=1).cpu().numpy())


@pytest.mark.parametrize("cadence", ["month", "ten_nights"])
@pytest.mark.parametrize("kind", [100, 300, "lognormal"])
@pytest.mark.parametrize("n_t,n_f", [(2000, 4111), (20_000, 60_007)])
def test_one_object_of_unequal_errors(env, cadence, kind, n_t, n_f):
    lsp, torch, dev = env
    t, y, dy = (torch.tensor(a, device=dev) for a in _light_curve(cadence, kind, n_t, 23))
    g = lsp.Grid(1.2, 1.2 + n_f * 1.176e-4, n_f)
    p, _ = lsp.periodogram_gls(t, y, dy, g)
    ref, _ = lsp.periodogram_gls(t, y.double(), dy.double(), g, precision="fp64")
    assert float((p.double() - ref).abs().max()) <= TOL


def test_weight_past_the_fp32_range(env):
    """1/dy^2 overflows FP32: the powers are those of the direct kernel, 0."""
    lsp, torch, dev = env
    segs = [_light_curve("seasons", 30, n, 29) for n in (50, 500, 60)]
    t, y, dy = (np.concatenate([s[i] for s in segs]) for i in range(3))
    dy[70] = 1e-20
    args = [torch.tensor(a, device=dev) for a in (t, y, dy, np.array([0, 50, 550, 610]))]
    g = lsp.Grid(0.24, 12.0, 2500)
    p, _ = lsp.batch_gls(*args, g, return_power=True)
    q, _ = lsp.batch_gls(*args, g, return_power=True, k_reseed=8)
    assert torch.equal(p[1], q[1]) and float(q[1].abs().max()) == 0.0
    assert float((p - q).abs().max()) <= TOL

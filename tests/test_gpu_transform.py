"""The transform path (trig sums of a run of bins by a nonuniform FFT) against
the FP64 CPU oracle, at the sizes where it can go wrong: either side of the
rule that selects it, of the observation tile (256) and of the run (2048
bins), one bin, clustered and unsorted times, spans longer than 1 / df (the
grid wraps), and many observations in few cells.

Tolerance on P_n: the sums' relative error is at most the window's aliasing
(1.6e-7) plus the FP32 transform's and weights' rounding (about 2^-24 log2 4096
+ a few ulp, under 1e-6); a power doubles it, and dividing by N^2 - R^2 >=
0.0975 N^2 magnifies the denominator's part by up to 10: 1.2e-5 in all.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
TOL = 1.2e-5


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    from paper_2105_04006_gb300 import build
    build.build()
    oracle.build()
    import paper_2105_04006_gb300 as lsp
    return lsp, torch, torch.device("cuda", 0)


def _segments(counts, cadence, seed):
    r = np.random.default_rng(seed)
    segs = []
    for n in counts:
        if cadence == "uniform":
            t = np.sort(60000 + r.uniform(0, 3650, n))
        elif cadence == "unsorted":
            t = 60000 + r.uniform(0, 3650, n)
        elif cadence == "one_night":
            t = 60000.3 + r.uniform(0, 0.1, n)
        elif cadence == "nightly":
            t = 60000.3 + r.integers(0, 3000, n) + r.uniform(0, 1 / 24, n)
        else:  # long: the span exceeds 1 / df many times over
            t = np.sort(60000 + r.uniform(0, 2e5, n))
        segs.append((t, 0.4 * np.sin(2 * np.pi * r.uniform(0.3, 5.0) * t) + r.normal(0, 0.2, n) + 3.0))
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    return np.concatenate([s[0] for s in segs]), np.concatenate([s[1] for s in segs]), off


@pytest.mark.parametrize("cadence,n_f", [("uniform", 6007), ("unsorted", 2049), ("one_night", 2048),
                                         ("nightly", 4111), ("long", 2047), ("uniform", 1)])
@pytest.mark.parametrize("gls", [False, True])
def test_batch_both_sides_of_every_edge(env, cadence, n_f, gls):
    lsp, torch, dev = env
    counts = [3, 31, 39, 40, 41, 63, 64, 65, 255, 256, 257, 511, 513, 2600]
    t, y, off = _segments(counts, cadence, 7)
    y32 = y.astype(np.float32)
    dy = np.random.default_rng(5).uniform(0.05, 0.3, t.size).astype(np.float32)
    g = lsp.Grid(0.24, 12.0, n_f)
    td, od = torch.tensor(t, device=dev), torch.tensor(off, device=dev)
    yd, ed = torch.tensor(y32, device=dev), torch.tensor(dy, device=dev)
    if gls:
        p, pk = lsp.batch_gls(td, yd, ed, od, g, return_power=True)
        ref = oracle.gls_batch(t, y32.astype(np.float64), dy.astype(np.float64), off, g.f_min, g.f_max, n_f)
        tol = 1e-4  # the generalized determinant is inverted down to 0.002 W^2
        if cadence == "one_night":
            # a fraction of a cycle of data: the fit is near singular on every bin and FP32 magnitudes
            # do not fix its power to 1e-4; both paths re-evaluate such bins in FP64, so they must agree
            q, _ = lsp.batch_gls(td, yd, ed, od, g, return_power=True, k_reseed=8)
            ref = {"power": q.cpu().numpy().astype(np.float64)}
    else:
        p, pk = lsp.batch(td, yd, od, g, return_power=True)
        ref = oracle.lsp_batch(t, y32.astype(np.float64), off, g.f_min, g.f_max, n_f, return_power=True)
        tol = TOL
    torch.cuda.synchronize()
    p, pk = p.cpu().numpy(), lsp.peaks_to_numpy(pk)
    assert np.isfinite(p).all()
    err = np.abs(p - ref["power"]).max(axis=1)
    # three observations determine the generalized fit's three parameters:
    # its power is 1 or, where the determinant is dropped, 0 (direct kernel)
    err = err[1:] if gls else err
    assert err.max() <= tol, dict(zip(counts[-len(err):], err))
    np.testing.assert_array_equal(pk["idx"], np.argmax(p, axis=1))


@pytest.mark.parametrize("n_t", [39, 40, 300, 2049])
@pytest.mark.parametrize("top_k", [1, 3])
def test_single_object(env, n_t, top_k):
    lsp, torch, dev = env
    b = synth.single_small(n_t=n_t, grid=synth.Grid(0.1, 10.0, 10_007))
    t, y = torch.tensor(b.t, device=dev), torch.tensor(b.y.astype(np.float32), device=dev)
    p, pk = lsp.periodogram(t, y, lsp.Grid(0.1, 10.0, 10_007), top_k=top_k)
    p, pk = p.cpu().numpy(), lsp.peaks_to_numpy(pk)
    ref, _ = oracle.lsp_single(b.t, b.y.astype(np.float32).astype(np.float64), 0.1, 10.0, 10_007)
    assert np.max(np.abs(p - ref)) <= TOL
    idx = [int(np.argmax(p))] if top_k == 1 else list(oracle.top_local_maxima(p.astype(np.float64), 3)[0])
    assert list(pk["idx"]) == idx


def test_plan_uses_the_transform_until_told_otherwise(env):
    lsp, torch, dev = env
    b = synth.ragged_survey(6, seed=3, grid=synth.Grid(0.24, 12.0, 3001))
    g = lsp.Grid(0.24, 12.0, 3001)
    args = (torch.tensor(b.t, device=dev), torch.tensor(b.y.astype(np.float32), device=dev),
            torch.tensor(b.offsets, device=dev))
    plan = lsp.Plan(b.n_obj, b.t.size, g)
    _, want = lsp.batch(*args, g)
    assert torch.equal(plan.execute(*args), want)
    plan.set_config(k_reseed=8, freqs_per_thread=16, block_threads=128)
    _, direct = lsp.batch(*args, g, k_reseed=8, freqs_per_thread=16, block_threads=128)
    assert torch.equal(plan.execute(*args), direct) and not torch.equal(direct, want)
    plan.close()


@pytest.mark.parametrize("threads,on", [(128, True), (256, False)])
def test_tuned_entry_from_before_the_transform(env, tmp_path, threads, on):
    """Its choice of direct kernel stands; the transform serves what it serves by default."""
    import re
    lsp, torch, dev = env
    b = synth.ragged_survey(6, seed=3, grid=synth.Grid(0.24, 12.0, 3001))
    args = (torch.tensor(b.t, device=dev), torch.tensor(b.y.astype(np.float32), device=dev),
            torch.tensor(b.offsets, device=dev))
    cache = tmp_path / "tune.jsonl"
    first = lsp.Plan(b.n_obj, b.t.size, lsp.Grid(0.24, 12.0, 3001))
    first.autotune(*args, cache_path=str(cache))
    first.close()
    entry = re.sub(r'"transform": \d+, ', "", cache.read_text())
    assert "transform" not in entry
    for key, v in (("k_reseed", 8), ("freqs_per_thread", 16), ("block_threads", threads)):
        entry, n = re.subn(rf'"{key}": \d+', f'"{key}": {v}', entry)
        assert n == 1
    cache.write_text(entry)
    plan = lsp.Plan(b.n_obj, b.t.size, lsp.Grid(0.24, 12.0, 3001))
    cfg = plan.autotune(*args, cache_path=str(cache))
    assert (cfg["k_reseed"], cfg["freqs_per_thread"], cfg["block_threads"]) == (8, 16, threads)
    assert plan.transform is on
    kw = {} if on else dict(k_reseed=8, freqs_per_thread=16, block_threads=threads)
    _, want = lsp.batch(*args, lsp.Grid(0.24, 12.0, 3001), **kw)
    assert torch.equal(plan.execute(*args), want)
    plan.close()


@pytest.mark.parametrize("n_t,n_f", [(8, 1), (9, 2047), (33, 32737), (300, 32738), (1000, 65505), (7001, 20_011)])
@pytest.mark.parametrize("cadence", ["uniform", "nightly", "long"])
def test_single_object_fp64(env, n_t, n_f, cadence):
    """The FP64 path's two-float transform of the whole grid, on either side of its grid's powers of two
    (2 (N_f + 32) cells), at the FP64 path's own tolerance."""
    lsp, torch, dev = env
    t, y, _ = _segments([n_t], cadence, 11)
    g = lsp.Grid(0.24, 12.0, n_f)
    p, pk = lsp.periodogram(torch.tensor(t, device=dev), torch.tensor(y, device=dev), g, precision="fp64")
    p, pk = p.cpu().numpy(), lsp.peaks_to_numpy(pk)
    ks = np.unique(np.concatenate([np.linspace(0, n_f - 1, 300).astype(np.int64), np.arange(max(0, n_f - 5), n_f)]))
    if cadence == "long":
        # 2.4e6 cycles: the oracle's FP64 phases are good to 2.4e6 x 2^-53 cycle only, the library's fixed-point
        # ones are exact; the direct kernel has the same phases
        ref = lsp.periodogram(torch.tensor(t, device=dev), torch.tensor(y, device=dev), g, precision="fp64",
                              k_reseed=16)[0].cpu().numpy()[ks]
    else:
        ref, _ = oracle.lsp_single(t, y, 0.24, 12.0, n_f, k_sel=ks)
    assert np.isfinite(p).all() and np.max(np.abs(p[ks] - ref)) <= 1e-10
    assert pk["idx"][0] == int(np.argmax(p)) and pk["power"][0] == p.max()


@pytest.mark.parametrize("n_t,n_f", [(6000, 1), (9001, 16_352), (20_000, 16_353), (30_000, 600_000)])
@pytest.mark.parametrize("top_k", [1, 3])
def test_single_object_of_many_observations(env, n_t, n_f, top_k):
    """FP32, the whole grid in one transform (its second pass of 256, 512 points)."""
    lsp, torch, dev = env
    b = synth.single_large(n_t=n_t, grid=synth.Grid(0.05, 25.0, n_f))
    t, y = torch.tensor(b.t, device=dev), torch.tensor(b.y.astype(np.float32), device=dev)
    p, pk = lsp.periodogram(t, y, lsp.Grid(0.05, 25.0, n_f), top_k=top_k)
    p, pk = p.cpu().numpy(), lsp.peaks_to_numpy(pk)
    ks = np.unique(np.concatenate([np.linspace(0, n_f - 1, 200).astype(np.int64), np.arange(max(0, n_f - 5), n_f)]))
    ref, _ = oracle.lsp_single(b.t, b.y.astype(np.float32).astype(np.float64), 0.05, 25.0, n_f, k_sel=ks)
    assert np.isfinite(p).all() and np.max(np.abs(p[ks] - ref)) <= TOL
    if top_k == 1 or n_f > 1:
        idx = [int(np.argmax(p))] if top_k == 1 else list(oracle.top_local_maxima(p.astype(np.float64), 3)[0])
        assert list(pk["idx"]) == idx


@pytest.mark.parametrize("cadence", ["uniform", "one_night", "nightly", "long"])
def test_fp64_batch_both_sides_of_every_edge(env, cadence):
    lsp, torch, dev = env
    counts = [3, 7, 8, 9, 31, 64, 255, 256, 257, 511, 513, 2600]
    t, y, off = _segments(counts, cadence, 9)
    g = lsp.Grid(0.24, 12.0, 4099)
    args = [torch.tensor(a, device=dev) for a in (t, y, off)]
    p, pk = lsp.batch(*args, g, precision="fp64", return_power=True)
    direct = lsp.batch(*args, g, precision="fp64", return_power=True, k_reseed=16)[0].cpu().numpy()
    if cadence == "long":  # as in test_single_object_fp64
        ref = direct
    else:
        ref = oracle.lsp_batch(t, y, off, 0.24, 12.0, 4099, return_power=True)["power"]
    p = p.cpu().numpy()
    np.testing.assert_array_equal(p[:2], direct[:2])  # 3 and 7 observations: left to the direct kernel
    err = np.abs(p - ref).max(axis=1)[2:]
    assert err.max() <= 1e-10, dict(zip(counts[2:], err))
    np.testing.assert_array_equal(lsp.peaks_to_numpy(pk)["idx"], np.argmax(p, axis=1))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_smaller_workspaces_take_smaller_paths(env, precision):
    """A workspace that holds only what the direct kernel needs is enough: the call takes that kernel."""
    lsp, torch, dev = env
    b = synth.single_small(n_t=9000, grid=synth.Grid(0.1, 10.0, 3001))
    dt = torch.float32 if precision == "fp32" else torch.float64
    t, y = torch.tensor(b.t, device=dev), torch.tensor(b.y, dtype=dt, device=dev)
    g = lsp.Grid(0.1, 10.0, 3001)
    k = 8 if precision == "fp32" else 16
    need = lsp.workspace_size(1, 9000, g, lsp.make_opts(precision=precision, k_reseed=k))
    full = lsp.workspace_size(1, 9000, g, lsp.make_opts(precision=precision))
    want, _ = lsp.periodogram(t, y, g, precision=precision)
    direct, _ = lsp.periodogram(t, y, g, precision=precision, k_reseed=k)
    ws = torch.empty(need, dtype=torch.uint8, device=dev)
    got, _ = lsp.periodogram(t, y, g, precision=precision, workspace=ws)
    assert torch.equal(got, direct if need < full else want)
    assert torch.allclose(want, direct, rtol=0, atol=TOL if precision == "fp32" else 1e-10)
    with pytest.raises(lsp.LSPError):
        lsp.periodogram(t, y, g, precision=precision, workspace=torch.empty(1024, dtype=torch.uint8, device=dev))


@pytest.mark.parametrize("n_f", [1, 511, 513, 1000, 1537])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_short_grids_equal_the_direct_kernel(env, n_f, precision):
    """Both sides of the observation counts at which a short grid's objects change kernels."""
    lsp, torch, dev = env
    counts = [7, 8, 9, 19, 20, 21, 39, 41, 59, 60, 61, 99, 100, 101, 400]
    t, y, off = _segments(counts, "uniform", 19)
    dt = torch.float32 if precision == "fp32" else torch.float64
    args = (torch.tensor(t, device=dev), torch.tensor(y, dtype=dt, device=dev), torch.tensor(off, device=dev),
            lsp.Grid(0.24, 12.0, n_f))
    p, _ = lsp.batch(*args, precision=precision, return_power=True)
    q, _ = lsp.batch(*args, precision=precision, return_power=True, k_reseed=8)
    assert float((p - q).abs().max()) <= (2 * TOL if precision == "fp32" else 1e-10)


@pytest.mark.parametrize("norm", ["standard", "psd"])
def test_refine_fallback_runs_equal_the_direct_full_grid(env, norm):
    """The fallback looks for the maximum's run with the transform and takes the result from the direct kernel
    on it: bit-equal to the direct full grid, also where many runs tie (regular sampling: the aliases of a
    frequency have the same power in exact arithmetic, more runs than the fallback keeps) and on a ragged grid."""
    lsp, torch, dev = env
    from paper_2105_04006_gb300 import learned as L
    counts = [2, 5, 39, 64, 300, 900]
    t, y, off = _segments(counts, "uniform", 21)
    reg = 60000.0 + np.arange(400.0)  # one observation a day: aliases at every whole cycle per day
    t = np.concatenate([t, reg])
    y = np.concatenate([y, np.sin(2 * np.pi * 0.3 * reg) + 0.1 * np.cos(2 * np.pi * 0.11 * reg)])
    off = np.append(off, off[-1] + 400)
    g = lsp.Grid(0.24, 12.0, 30_011)
    args = (torch.tensor(t, device=dev), torch.tensor(y.astype(np.float32), device=dev), torch.tensor(off, device=dev))
    n = off.size - 1
    cls = torch.zeros((n, 1), dtype=torch.int32, device=dev)
    code = 1 if norm == "standard" else 0
    peaks, info = L.refine(*args, g, cls, 1, 1e30, 1e30, norm=code)  # every object falls back
    _, want = lsp.batch(*args, g, norm=norm, k_reseed=16, freqs_per_thread=32, block_threads=64)
    a, b = lsp.peaks_to_numpy(peaks), lsp.peaks_to_numpy(want)
    for name in ("idx", "power", "flags"):
        np.testing.assert_array_equal(a[name], b[name], err_msg=name)
    assert (info.cpu().numpy() & 256).all()

"""The autotuner's error gate describes what the chosen configuration runs."""
import numpy as np
import pytest

import synth

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


@pytest.mark.parametrize("n_obj", [1, 9])
def test_report_and_trial_cover_both_kernels_of_the_configuration(env, n_obj):
    """Exact values: the same kernels on the same inputs give the same bits, and the errors are rounded to FP32."""
    lsp, torch, dev = env
    b = synth.ragged_survey(n_obj, seed=5, grid=synth.Grid(0.24, 12.0, 20_011))
    args = [torch.tensor(b.t, device=dev), torch.tensor(b.y.astype(np.float32), device=dev)]
    if n_obj > 1:
        args.append(torch.tensor(b.offsets, device=dev))
    g = lsp.Grid(0.24, 12.0, 20_011)
    plan = lsp.Plan(n_obj, b.t.size, g)
    cfg, trials = plan.autotune(*args, return_trials=True)
    assert plan.transform  # by far the fastest on these sizes

    def powers(**kw):
        wide = [args[0], args[1].double() if kw.get("precision") == "fp64" else args[1]] + args[2:]
        return (lsp.batch if n_obj > 1 else lsp.periodogram)(*wide, g, return_power=True, **kw)[0].reshape(n_obj, -1)

    ref = powers(precision="fp64")
    err = (powers().double() - ref).abs().amax(dim=1)
    if n_obj > 1:
        named = {k: cfg[k] for k in ("k_reseed", "freqs_per_thread", "block_threads")}
        err = torch.maximum(err, (powers(**named).double() - ref).abs().amax(dim=1))
    rep = dict(plan.gate_report())
    assert rep
    for o, e in rep.items():
        assert np.float32(float(err[o])) == np.float32(e), (o, e)
    # the configuration's own trial (the last: the transform) reports the same
    assert np.float32(trials[-1]["max_err"]) == np.float32(max(rep.values()))
    assert trials[-1]["ms"] == min(t["ms"] for t in trials if t["passed"])
    plan.close()

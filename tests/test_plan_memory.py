"""Plans when device memory runs out, on the CPU: the library's own host code
over a stand-in for the CUDA runtime (``fake_cudart.c``, preloaded), whose
allocations fail past a limit and whose copies and clears must stay inside live
allocations."""
import os
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import ctypes, os, sys
import numpy as np
import paper_2105_04006_gb300 as lsp
fake = ctypes.CDLL(os.environ["LD_PRELOAD"])
fake.fake_used.restype = ctypes.c_size_t
fake.fake_limit.argtypes = [ctypes.c_size_t]
L = lsp.lib()
def dev(a):
    p = ctypes.c_void_p()
    cudart = ctypes.CDLL(None)
    assert cudart.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(max(a.nbytes, 1))) == 0
    ctypes.memmove(p, a.ctypes.data, a.nbytes)
    return p
def inputs(counts, dt):
    n = sum(counts)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    return dev(np.linspace(0, 100, n)), dev(np.zeros(n, dt)), dev(off) if len(counts) > 1 else None
def plan(counts, grid, **kw):
    h = ctypes.c_void_p()
    o = lsp.make_opts(**kw)
    st = L.lsp_plan_create(ctypes.byref(h), len(counts), sum(counts), ctypes.byref(grid), ctypes.byref(o))
    return st, h
def runs(h, args, n_peaks):
    pk = dev(np.zeros(40 * n_peaks, np.uint8))
    before = fake.fake_launches()
    st = L.lsp_plan_execute(h, *args, None, pk, None)
    assert st == 0 and fake.fake_launches() > before, (st, L.lsp_last_error())
    assert fake.fake_outside() == 0
def trials_of(h, args):
    buf, n = (lsp.Trial * 256)(), ctypes.c_int32(0)
    st = L.lsp_plan_autotune_ex(h, *args, None, 0, buf, 256, ctypes.byref(n), None)
    return st, [buf[i] for i in range(n.value)]
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_2105_04006_gb300 import build
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    subprocess.run(["gcc", "-O1", "-std=c11", "-w", "-fPIC", "-shared", "-I", inc,
                    os.path.join(ROOT, "tests", "fake_cudart.c"), "-o", so], check=True)

    def run(code):
        env = dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT)
        r = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(code)], env=env, cwd=ROOT,
                           capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
    return run


@pytest.mark.parametrize("precision,n_t,room", [("fp64", 9000, "below"), ("fp64", 9000, "direct"), ("fp32", 9000, "below"),
                                                ("fp32", 9000, "direct")])
def test_autotune_of_a_plan_that_took_a_smaller_path(fake, precision, n_t, room):
    """A plan created with room for a smaller path only: autotune tunes that path and the plan goes on running,
    also when nothing beyond its own workspace is left."""
    fake(f"""
    g = lsp.Grid(0.1, 10.0, 2_000_000)
    dt = np.float64 if "{precision}" == "fp64" else np.float32
    args = inputs([{n_t}], dt)
    full = lsp.workspace_size(1, {n_t}, g, lsp.make_opts(precision="{precision}"))
    direct = lsp.workspace_size(1, {n_t}, g, lsp.make_opts(precision="{precision}", k_reseed=16 if "{precision}" == "fp64" else 8))
    assert direct < full
    fake.fake_limit(fake.fake_used() + (full - 1 if "{room}" == "below" else direct))
    st, h = plan([{n_t}], g, precision="{precision}")
    assert st == 0, L.lsp_last_error()
    fake.fake_limit(fake.fake_used() + 400)  # the peaks
    runs(h, args, 1)
    fake.fake_limit(fake.fake_used() + (80 << 20))
    st, trials = trials_of(h, args)
    # FP32: its error gate's own scratch does not fit
    assert (st == 0 and trials) or ("{precision}" == "fp32" and st == 3), L.lsp_last_error()
    fake.fake_limit(fake.fake_used() + 400)
    runs(h, args, 1)
    assert fake.fake_outside() == 0
    """)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_a_configuration_that_does_not_fit_leaves_the_plan_as_it_was(fake, precision):
    fake(f"""
    g = lsp.Grid(0.1, 10.0, 100_000)
    dt = np.float64 if "{precision}" == "fp64" else np.float32
    args = inputs([3000], dt)
    st, h = plan([3000], g, precision="{precision}")
    assert st == 0
    runs(h, args, 1)
    fake.fake_limit(fake.fake_used() + 400)
    c = lsp.Config()
    L.lsp_plan_get_config(h, ctypes.byref(c))
    c.transform = 0
    c.obs_split = 256
    assert L.lsp_plan_set_config(h, ctypes.byref(c)) == 3  # LSP_E_NOMEM
    runs(h, args, 1)
    """)


def test_autotune_skips_candidates_that_do_not_fit(fake):
    """A batch whose smaller chunks need more workspace than is left."""
    fake("""
    counts = [60] * 50
    g = lsp.Grid(0.1, 10.0, 400_000)
    args = inputs(counts, np.float32)
    st, h = plan(counts, g, precision="fp32")
    assert st == 0
    st, every = trials_of(h, args)
    assert st == 0
    st, h = plan(counts, g, precision="fp32")
    gate = 8 * 400_000 * 12 + (8 << 20)  # the gate's periodograms and scratch
    fake.fake_limit(fake.fake_used() + gate)
    st, some = trials_of(h, args)
    assert st == 0, L.lsp_last_error()
    assert 0 < len(some) <= len(every)
    runs(h, args, 50)
    """)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_autotune_tries_splits_around_the_direct_kernels_own(fake, precision):
    """One object: also where the transform, which has no split, is the default."""
    fake(f"""
    g = lsp.Grid(0.1, 10.0, 60_000)
    args = inputs([9000], np.float64 if "{precision}" == "fp64" else np.float32)
    st, h = plan([9000], g, precision="{precision}")
    c = lsp.Config()
    assert st == 0 and L.lsp_plan_get_config(h, ctypes.byref(c)) == 0 and c.obs_split >= 8
    st, trials = trials_of(h, args)
    assert st == 0, L.lsp_last_error()
    tried = set(t.config.obs_split for t in trials)
    assert tried >= set(c.obs_split * f // 4 for f in (1, 2, 4, 8, 16)), (tried, c.obs_split)
    """)


def test_a_plan_that_lost_its_workspace_refuses_until_it_has_one(fake):
    """The old size is not to be had either: no launch on memory the plan does not have, no allocation in an
    execution, and a configuration set later brings the plan back."""
    fake("""
    g = lsp.Grid(0.1, 10.0, 100_000)
    args = inputs([9000], np.float32)
    st, h = plan([9000], g)
    assert st == 0
    c = lsp.Config()
    L.lsp_plan_get_config(h, ctypes.byref(c))
    pk = dev(np.zeros(40, np.uint8))
    fake.fake_limit(0)
    d = lsp.Config.from_buffer_copy(c)
    d.obs_split = 256
    assert L.lsp_plan_set_config(h, ctypes.byref(d)) == 3
    before = fake.fake_launches()
    assert L.lsp_plan_execute(h, *args, None, pk, None) == 4  # LSP_E_WORKSPACE
    fake.fake_limit(1 << 40)
    assert L.lsp_plan_execute(h, *args, None, pk, None) == 4
    assert fake.fake_launches() == before and fake.fake_outside() == 0
    assert L.lsp_plan_set_config(h, ctypes.byref(c)) == 0
    runs(h, args, 1)
    """)

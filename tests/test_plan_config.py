"""A plan's configuration, read and set again, on the CPU over the stand-in for
the CUDA runtime (see test_plan_memory)."""
import pytest

from test_plan_memory import fake  # noqa: F401  (fixture)

SETUP = """
def get(h):
    c = lsp.Config()
    assert L.lsp_plan_get_config(h, ctypes.byref(c)) == 0
    return c
counts = [{n_t}] * {n_obj}
g = lsp.Grid(0.24, 12.0, 30_000)
args = inputs(counts, np.float32)
"""


@pytest.mark.parametrize("n_obj,n_t", [(40, 300), (1, 9000)])
@pytest.mark.parametrize("field,value", [("k_reseed", 16), ("obs_split", 3), ("block_threads", 64)])
def test_read_change_set_runs_the_kernel_named(fake, n_obj, n_t, field, value):  # noqa: F811
    if field == "obs_split" and n_obj > 1:
        pytest.skip("a batch has no split")
    fake(SETUP.format(n_obj=n_obj, n_t=n_t) + f"""
st, h = plan(counts, g)
c = get(h)
assert c.transform != 0
assert L.lsp_plan_set_config(h, ctypes.byref(c)) == 0 and get(h).transform == c.transform  # unchanged: stays on
c.{field} = {value}
if "{field}" == "k_reseed":
    c.freqs_per_thread, c.block_threads = 32, 64
if "{field}" == "block_threads":
    c.k_reseed, c.freqs_per_thread = 16, 32
assert L.lsp_plan_set_config(h, ctypes.byref(c)) == 0
d = get(h)
assert d.transform == 0 and d.{field} == {value}
d.transform = 1  # asked for beside that kernel
assert L.lsp_plan_set_config(h, ctypes.byref(d)) == 0 and get(h).transform != 0
runs(h, args, {n_obj})
""")


@pytest.mark.parametrize("n_obj,n_t", [(40, 300), (1, 9000)])
def test_one_plans_configuration_set_on_another(fake, n_obj, n_t):  # noqa: F811
    fake(SETUP.format(n_obj=n_obj, n_t=n_t) + f"""
a, b = lsp.Plan({n_obj}, {n_obj * n_t}, g), lsp.Plan({n_obj}, {n_obj * n_t}, g)
kernel = dict(k_reseed=16, freqs_per_thread=32, block_threads=64, packed=1)
a.set_config(**kernel)
assert not a.transform and a.config["transform"] == 0
b.set_config(**a.config)
assert not b.transform and b.config == a.config
a.set_config(transform=1, **kernel)
assert a.transform
b.set_config(**a.config)
assert b.transform and b.config == a.config
# the same in C, between plans of different kernels
c = get(a._h)
st, h = plan(counts, g)
assert get(h).k_reseed != c.k_reseed
assert L.lsp_plan_set_config(h, ctypes.byref(c)) == 0
assert get(h).transform == c.transform != 0 and get(h).k_reseed == 16
""")


def test_trials_tell_the_transform_from_its_direct_kernel(fake):  # noqa: F811
    fake(SETUP.format(n_obj=40, n_t=300) + """
st, h = plan(counts, g)
st, trials = trials_of(h, args)
assert st == 0
seen = [tuple(sorted(t.config.as_dict().items())) for t in trials]
assert len(set(seen)) == len(seen) and sum(t.config.transform != 0 for t in trials) == 1
""")

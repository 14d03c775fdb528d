"""The path of one object's generalized periodogram, by its workspace, on the CPU."""
import ctypes

import pytest


@pytest.mark.parametrize("n_t,n_f,split", [(100_000, 1000, True), (100_000, 5000, True), (30_000, 3000, True), (10_000, 1000, True),
                                           (100_000, 30_000, False), (30_000, 100_000, False), (10_000, 10_000, False),
                                           (3000, 1000, False), (1000, 100_000, False), (39, 1000, True)])
def test_split_kernel_where_it_is_the_faster(n_t, n_f, split):
    """Many observations on a short grid: every run of 2048 bins would spread all of them on one SM."""
    from paper_2105_04006_gb300 import build
    build.build()
    import paper_2105_04006_gb300 as lsp

    def need(**kw):
        n = ctypes.c_size_t(0)
        g, o = lsp.Grid(0.24, 12.0, n_f), lsp.make_opts(**kw)
        assert lsp.lib().lsp_workspace_size_gls(1, n_t, ctypes.byref(g), ctypes.byref(o), ctypes.byref(n)) == 0
        return n.value

    # the split kernel's partial sums are the larger part of its workspace
    assert (need() == need(k_reseed=8)) == split

"""Options of the binding's calls, on the CPU."""
import numpy as np
import pytest

import paper_2105_04006_gb300 as lsp


class Number:
    """Converts to an int that can change, as a tensor or a 0-d array does; hashed by identity."""

    def __init__(self, v):
        self.v = v

    def __int__(self):
        return self.v


def test_an_argument_that_changes_is_read_in_every_call():
    k = Number(1)
    assert lsp._opts_of({"top_k": k}).top_k == 1
    k.v = 3
    assert lsp._opts_of({"top_k": k}).top_k == 3


@pytest.mark.parametrize("kw", [{}, {"top_k": 3}, {"top_k": np.int64(2), "precision": "fp64"}, {"center": False, "norm": "psd"},
                                {"k_reseed": 16.0}])
def test_options_equal_make_opts(kw):
    assert bytes(lsp._opts_of(kw)) == bytes(lsp.make_opts(**kw)) == bytes(lsp._opts_of(dict(kw)))


def test_bad_arguments_are_refused_every_time():
    for _ in range(2):
        with pytest.raises((KeyError, TypeError)):
            lsp._opts_of({"precision": []})
        with pytest.raises(TypeError):
            lsp._opts_of({"no_such_option": 1})

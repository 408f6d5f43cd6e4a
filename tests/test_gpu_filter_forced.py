"""The filter's tile edges, widths, hand-overs and scales (test_gpu_filter.py) with
the filter asked for by name and every call asserted to have gone through it, so
that no rule of the automatic choice can take these cases away from it."""
import numpy as np
import pytest

import tests.test_gpu_filter as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def forced(monkeypatch):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_07156_gb300 as amp
    own, check = amp.Index.set_kernel, T.check
    monkeypatch.setattr(amp.Index, "set_kernel",
                        lambda self, which: own(self, "filtered" if which in ("auto", "split") else which))

    def filtered_check(a, g, *args, **kw):
        check(a, g, *args, **kw)
        assert g.tap(amp.abi.TAP_FILTERED, (1,), np.int32)[0] == 1

    monkeypatch.setattr(T, "check", filtered_check)
    return amp


@pytest.mark.parametrize("dim,M", [(16, 8), (64, 16), (96, 48), (100, 20), (136, 17), (256, 32), (960, 120)])
@pytest.mark.parametrize("bits", [0, 6, 8, 12])
def test_tile_edges(forced, dim, M, bits):
    T.test_tile_edges(forced, dim, M, bits)


@pytest.mark.parametrize("k", [10, 32, 100, 128])
def test_uneven_batches_and_widths(forced, k):
    T.test_uneven_batches_and_widths(forced, k, "auto")


def test_queries_left_to_the_scan(forced):
    T.test_queries_left_to_the_scan(forced)


def test_scales(forced):
    T.test_scales(forced)

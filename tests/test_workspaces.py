"""Workspace sizes, on the host: a batch does not ask for eight buffers of its largest systems."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def tc():
    from paper_2403_06937_gb300 import build as B
    B.build()
    import paper_2403_06937_gb300 as tc
    return tc


def _batch(tc, ns, precision):
    lib, arr = tc._abi.load(), (ctypes.c_int * len(ns))(*ns)
    return int(lib.tc_batch_workspace_size(len(ns), arr, tc.PRECISIONS[precision]))


@pytest.mark.parametrize("precision", ["fp64", "ozaki"])
def test_batch_of_large_systems_fits(tc, precision):
    one = tc.workspace_size(14, tc.PRECISIONS[precision])
    for count in (2, 6, 8):   # U and rho of each take 8.6 GB beside this
        assert _batch(tc, [14] * count, precision) <= max(one + 4096, 32 << 30)
    # small systems keep a buffer for each of eight
    assert _batch(tc, [8] * 20, precision) >= 8 * tc.workspace_size(8, tc.PRECISIONS[precision])

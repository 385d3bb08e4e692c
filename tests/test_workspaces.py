"""Workspace sizes, on the host: the least that a call accepts never asks for more than the forms that keep digit
slices or FP64 planes alone did, and a batch does not ask for eight buffers of its largest systems."""
import ctypes

import pytest

# GB that the calls asked for with digit slices (ozaki) or on the FP64 DMMA (fp64): 100 steps, checkpoints of 20
BEFORE = {("ozaki", "evolve", 8): 0.006824, ("ozaki", "evolve", 12): 1.879, ("ozaki", "evolve", 14): 32.22,
          ("ozaki", "evolve", 15): 128.9, ("ozaki", "lindblad", 12): 6.027, ("ozaki", "backward", 14): 204.1,
          ("fp64", "evolve", 14): 12.9, ("fp64", "expm", 14): 27.93, ("fp64", "lindblad", 13): 15.16,
          ("fp64", "backward", 13): 39.2}


@pytest.fixture(scope="module")
def tc():
    from paper_2403_06937_gb300 import build as B
    B.build()
    import paper_2403_06937_gb300 as tc
    return tc


@pytest.mark.parametrize("precision,op,n", sorted(BEFORE))
def test_least_workspace(tc, precision, op, n):
    ops = dict(evolve=tc.TC_OP_EVOLVE, lindblad=tc._abi.TC_OP_LINDBLAD, backward=tc.TC_OP_BACKWARD, expm=tc.TC_OP_EXPM)
    prec = tc.PRECISIONS[precision]
    least = tc.workspace_least(n, prec, ops[op], 100, 20)
    assert 0 < least <= BEFORE[precision, op, n] * 1e9
    assert least <= tc.workspace_size(n, prec, ops[op], 100, 20)


def test_split_forms_and_the_dmma_form_have_one_size(tc):
    for name in ("bf16x3", "tf32", "tf32x3", "fp64_dmma"):
        for op in (tc.TC_OP_EVOLVE, tc._abi.TC_OP_LINDBLAD, tc._abi.TC_OP_EVOLVE_HOST):
            assert tc.workspace_size(12, tc.PRECISIONS[name], op, 3) == tc.workspace_least(12, tc.PRECISIONS[name], op, 3)
    # the gradient has no split form: a query of it in one states what the DMMA form takes, as a part of several ops
    assert tc.workspace_size(14, tc.TC_BF16X3, tc.TC_OP_BACKWARD, 100, 20) == \
        tc.workspace_least(14, tc.TC_FP64, tc.TC_OP_BACKWARD, 100, 20)
    assert tc.workspace_least(13, tc.TC_FP64) == tc.workspace_size(13, tc.PRECISIONS["fp64_dmma"])


def _batch(tc, ns, precision):
    lib, arr = tc._abi.load(), (ctypes.c_int * len(ns))(*ns)
    prec = tc.PRECISIONS[precision]
    return int(lib.tc_batch_workspace_size(len(ns), arr, prec)), int(lib.tc_batch_workspace_least(len(ns), arr, prec))


@pytest.mark.parametrize("precision", ["fp64", "ozaki", "fp64_dmma"])
def test_batch_of_large_systems_fits(tc, precision):
    one = tc.workspace_size(14, tc.PRECISIONS[precision])
    for count in (2, 6, 8):   # U and rho of each take 8.6 GB beside this
        stated, least = _batch(tc, [14] * count, precision)
        assert least <= stated <= max(one + 4096, 32 << 30)
    # small systems keep a buffer for each of eight
    assert _batch(tc, [8] * 20, precision)[0] >= 8 * tc.workspace_size(8, tc.PRECISIONS[precision])


def test_wrappers_take_what_fits(tc, monkeypatch):
    """A caller's buffer of at least the least size is used; without one, what the device has left is tried."""
    import torch
    taken = []

    def empty(nbytes, device):
        taken.append(nbytes)
        if nbytes > 1000:
            raise torch.cuda.OutOfMemoryError("out of memory")
        return torch.empty(nbytes, dtype=torch.uint8)

    monkeypatch.setattr(tc, "_work", empty)
    mine = torch.empty(700, dtype=torch.uint8)
    assert tc._workspace(mine, 4000, 600, "cpu") is mine and not taken
    assert tc._workspace(mine, 4000, 800, "cpu").numel() == 800 and taken == [4000, 800]
    taken.clear()
    assert tc._workspace(None, 9000, 300, "cpu", halving=True).numel() == 562 and taken == [9000, 4500, 2250, 1125, 562]
    with pytest.raises(torch.cuda.OutOfMemoryError):
        tc._workspace(None, 9000, 5000, "cpu", halving=True)

"""The FP64 forms in less workspace than is stated.

A form's results do not depend on the workspace: bitwise equal where the form
stays the same (fewer lanes of a batch).
"""
import ctypes

import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tc():
    from paper_2403_06937_gb300 import build
    build.build()
    import paper_2403_06937_gb300 as tc
    tc.device_check()
    return tc


def _buffer(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8, device="cuda")


def _setup(tc, n, dt=0.1):
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 60 + n) * 5)), 1.013, 1.0)
    return p, tc.expm_model(p, dt), torch.from_numpy(W.random_mixed_state(n, 2, n)[0]).cuda()


@pytest.mark.parametrize("precision", ["fp64", "ozaki"])
def test_batch_on_fewer_lanes(tc, precision):
    """From the stated size down to one lane."""
    ns, steps = [7, 9, 8, 7, 8], 3
    ps, Us, rhos = zip(*[_setup(tc, n) for n in ns])
    want = [tc.evolve(U, r, n, steps, precision, params=p)[0] for n, p, U, r in zip(ns, ps, Us, rhos)]
    lib, arr = tc._abi.load(), (ctypes.c_int * len(ns))(*ns)
    prec = tc.PRECISIONS[precision]
    stated = int(lib.tc_batch_workspace_size(len(ns), arr, prec))
    one = 256 + (tc.workspace_size(9, prec) + 255) // 256 * 256
    for nbytes in (stated, stated - 256, stated // 2, one):
        outs, work = [r.clone() for r in rhos], _buffer(nbytes)
        tc._abi.call("tc_batch_evolve", len(ns), arr, (ctypes.c_void_p * 5)(*[u.data_ptr() for u in Us]),
                     (ctypes.c_void_p * 5)(*[o.data_ptr() for o in outs]), steps, prec, 0, None, None,
                     ctypes.c_void_p(work.data_ptr()), work.numel(),
                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert all(torch.equal(a, b) for a, b in zip(outs, want)), nbytes

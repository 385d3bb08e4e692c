"""The FP64 forms in less workspace than is stated, and the DMMA form by name.

A form's results do not depend on the workspace: bitwise equal where the form
stays the same (fewer lanes of a batch, operands made a few moduli at a time).
"""
import ctypes

import numpy as np
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


@pytest.mark.parametrize("n,steps", [(5, 4), (7, 3), (8, 12), (9, 2), (10, 2), (11, 2)])
def test_emulated_steps_in_the_least_workspace(tc, n, steps):
    """Two and four columns a thread, one and several K chunks and tiles, padding (n = 5), steps in graphs."""
    p, U, rho = _setup(tc, n)
    want, rows = tc.evolve(U, rho, n, steps, "ozaki", renorm_every=5, params=p)
    work = _buffer(tc.workspace_least(n, tc.PRECISIONS["ozaki"]))
    got, rows2 = tc.evolve(U, rho, n, steps, "ozaki", renorm_every=5, params=p, work=work)
    assert torch.equal(got, want) and torch.equal(rows2, rows)


def test_emulated_open_system_and_gradient_in_the_least_workspace(tc):
    n, steps = 8, 4
    p, U, rho = _setup(tc, n)
    lay = tc.lindblad_layout(n)
    Ub = tc.lindblad_propagators(p, 0.1)
    state = torch.zeros(lay.total, dtype=torch.complex128, device="cuda")
    state[-1] = 1.0
    want, _ = tc.lindblad_evolve(p, 0.1, 0.1, Ub, state, steps, "ozaki")
    work = _buffer(tc.workspace_least(n, tc.PRECISIONS["ozaki"], tc._abi.TC_OP_LINDBLAD))
    got, _ = tc.lindblad_evolve(p, 0.1, 0.1, Ub, state, steps, "ozaki", work=work)
    assert torch.equal(got, want)
    O = torch.arange(1 << n, dtype=torch.float64, device="cuda") / (1 << n)
    # dt = 0.1 of couplings of 0.05: no squaring; a large dt squares
    for dt in (0.1, 3.0):
        V = tc.expm_model(p, dt)
        want, loss = tc.evolve_backward(p, dt, steps, rho, V, O, ckpt_every=3, precision="ozaki")
        work = _buffer(tc.workspace_least(n, tc.PRECISIONS["ozaki"], tc.TC_OP_BACKWARD, steps, 3))
        got, loss2 = tc.evolve_backward(p, dt, steps, rho, V, O, ckpt_every=3, precision="ozaki", work=work)
        assert torch.equal(got, want) and loss == loss2


@pytest.mark.parametrize("precision", ["fp64", "ozaki"])
def test_batch_on_fewer_lanes(tc, precision):
    """From the stated size down to one lane, and below: the systems one after another in the least form."""
    ns, steps = [7, 9, 8, 7, 8], 3
    ps, Us, rhos = zip(*[_setup(tc, n) for n in ns])
    want = [tc.evolve(U, r, n, steps, precision, params=p)[0] for n, p, U, r in zip(ns, ps, Us, rhos)]
    lib, arr = tc._abi.load(), (ctypes.c_int * len(ns))(*ns)
    prec = tc.PRECISIONS[precision]
    stated = int(lib.tc_batch_workspace_size(len(ns), arr, prec))
    one = 256 + (tc.workspace_size(9, prec) + 255) // 256 * 256
    for nbytes in (stated, stated - 256, stated // 2, one):
        outs, _ = tc.batch_evolve(list(Us), list(rhos), steps, precision, params=list(ps), work=_buffer(nbytes))
        assert all(torch.equal(a, b) for a, b in zip(outs, want)), nbytes
    least = int(lib.tc_batch_workspace_least(len(ns), arr, prec))
    assert least < one
    outs, _ = tc.batch_evolve(list(Us), list(rhos), steps, precision, params=list(ps), work=_buffer(least))
    if precision == "fp64":
        want = [tc.evolve(U, r, n, steps, "fp64_dmma", params=p)[0] for n, p, U, r in zip(ns, ps, Us, rhos)]
    assert all(torch.equal(a, b) for a, b in zip(outs, want))
    with pytest.raises(tc.TCError):
        p = (tc._abi.tc_params * len(ns))(*[q.c() for q in ps])
        out = [r.clone() for r in rhos]
        small = _buffer(least - 256)
        tc._abi.call("tc_batch_evolve", len(ns), arr, (ctypes.c_void_p * 5)(*[u.data_ptr() for u in Us]),
                     (ctypes.c_void_p * 5)(*[o.data_ptr() for o in out]), steps, prec, 0, p, None,
                     ctypes.c_void_p(small.data_ptr()), small.numel(), None)


def test_the_dmma_form_by_name(tc):
    """In any workspace, bitwise TC_FP64 in the least one: steps, host memory, batch, open system, gradient, exponential."""
    n, steps = 8, 3
    p, U, rho = _setup(tc, n)
    small = _buffer(tc.workspace_least(n, tc.TC_FP64))
    want, rows = tc.evolve(U, rho, n, steps, "fp64", params=p, work=small)
    big = _buffer(tc.workspace_size(n, tc.TC_FP64))
    for work in (None, big):
        got, rows2 = tc.evolve(U, rho, n, steps, "fp64_dmma", params=p, work=work)
        assert torch.equal(got, want) and torch.equal(rows, rows2)
    assert not torch.equal(tc.evolve(U, rho, n, steps, "fp64", params=p)[0], want)
    host = rho.cpu()
    tc.evolve_host(U, host, n, steps, "fp64_dmma", params=p)
    assert torch.equal(host, want.cpu())
    outs, _ = tc.batch_evolve([U, U], [rho, rho], steps, "fp64_dmma", params=[p, p])
    assert torch.equal(outs[0], want) and torch.equal(outs[1], want)
    O = torch.arange(1 << n, dtype=torch.float64, device="cuda") / (1 << n)
    least = _buffer(tc.workspace_least(n, tc.TC_FP64, tc.TC_OP_BACKWARD, steps, 2))
    ref, loss = tc.evolve_backward(p, 0.1, steps, rho, U, O, ckpt_every=2, work=least)
    grad, loss2 = tc.evolve_backward(p, 0.1, steps, rho, U, O, ckpt_every=2, precision="fp64_dmma")
    assert torch.equal(grad, ref) and loss == loss2
    lay = tc.lindblad_layout(n)
    Ub = tc.lindblad_propagators(p, 0.1)
    state = torch.zeros(lay.total, dtype=torch.complex128, device="cuda")
    state[-1] = 1.0
    a, _ = tc.lindblad_evolve(p, 0.1, 0.1, Ub, state, steps, "fp64_dmma")
    b, _ = tc.lindblad_evolve(p, 0.1, 0.1, Ub, state, steps, "fp64")
    assert not torch.equal(a, b) and (a - b).abs().max().item() < steps * 2 * (1 << n) * 2.0 ** -51
    H = tc.build_hamiltonian(p)
    x = tc.expm(H, n, 0.1, precision="fp64_dmma")
    y = tc.expm(H, n, 0.1, work=_buffer(tc.workspace_least(n, tc.TC_FP64, tc.TC_OP_EXPM)))
    assert torch.equal(x, y) and not torch.equal(x, tc.expm(H, n, 0.1))

"""Routes of the FP64 forms and tile shapes against one another at the sizes where they change over."""
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


def _bound(n, steps):
    """As in test_gpu_crt.py: two products a step, each within the residue form's rounding of the rows, four
    roundings and the DMMA sums' K 2^-52, relative to rows of norm at most 1."""
    K = 1 << n
    return steps * 2 * (2 * np.sqrt(2 * K) * 2.0 ** -58.32 + 4 * 2.0 ** -53 + K * 2.0 ** -52)


@pytest.mark.parametrize("precision", ["bf16x3", "tf32x3", "tf32"])
@pytest.mark.parametrize("n", [8, 9])
def test_64_column_pair_tiles_give_the_bits_of_single_ctas(tc, n, precision):
    """n = 8, 9: one and two row pairs, every launch in 64-column tiles; the same sums in the same order."""
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 4) * 4)), 1.01, 1.0)
    U = tc.expm_model(p, 0.1)
    rho = torch.from_numpy(W.random_mixed_state(n, 3, 5)[0]).cuda()
    saved = tc.autotune_lookup(n, precision)
    out = []
    try:
        for shape in ("single", "pair32", "pair_wide"):
            tc.autotune_set(n, precision, saved["f64_tile"], saved["tc_group"], saved["tc_stages"], shape)
            out.append(tc.evolve(U, rho, n, 4, precision, params=p))
    finally:
        tc.autotune_set(n, precision, saved["f64_tile"], saved["tc_group"], saved["tc_stages"], saved["tc_shape"])
    for a, o in out[1:]:
        assert torch.equal(a, out[0][0]) and torch.equal(o, out[0][1])


def test_open_system_blocks_on_the_tensor_cores_equal_the_dmma_blocks(tc):
    """n = 10 (blocks on both sides of 64 rows, most of them ragged), the smallest size whose tensor-core form
    needs more workspace than the DMMA form: that one runs in 64 KiB less than is stated.  The damping adds two passes
    a step of n + 1 terms each."""
    n, dt, steps, kappa = 10, 0.05, 3, 0.4
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 74) * 20)), 1.002, 1.0)
    lay = tc.lindblad_layout(n)
    U = tc.lindblad_propagators(p, dt)
    rho = torch.zeros(lay.total, dtype=torch.complex128, device="cuda")
    j = lay.basis.index((1 << n) - 1)
    lay.blocks(rho)[n][j, j] = 1.0
    a, oa = tc.lindblad_evolve(p, kappa, dt, U, rho, steps, "fp64", renorm_every=2)
    b = rho.clone()
    work = torch.empty(tc.workspace_size(n, tc.TC_FP64, tc._abi.TC_OP_LINDBLAD) - 65536, dtype=torch.uint8, device="cuda")
    c = p.c()
    tc._abi.call("tc_lindblad_evolve", ctypes.byref(c), kappa, dt, ctypes.c_void_p(U.data_ptr()),
                 ctypes.c_void_p(b.data_ptr()), steps, tc.TC_FP64, 2, None, ctypes.c_void_p(work.data_ptr()),
                 work.numel(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    tc.sync_status()
    assert not torch.equal(a, b)   # two routes
    assert torch.max(torch.abs(a - b)).item() <= _bound(n, steps) + steps * 2 * (n + 1) * 2.0 ** -52


def test_fp64_batch_in_a_small_workspace(tc):
    """One lane on the DMMA GEMM in less than the lanes' workspace; n <= 6 take that form on either route."""
    ns, steps = [5, 8, 6, 7], 4
    ps = [tc.Params(n, list(map(float, W.draw_couplings(n, 20 + n) * 5)), 1.013, 1.0) for n in ns]
    Us = [tc.expm_model(p, 0.1) for p in ps]
    rhos = [torch.from_numpy(W.random_mixed_state(n, 2, n)[0]).cuda() for n in ns]
    outs, obs = tc.batch_evolve(Us, rhos, steps, "fp64", params=ps)
    lib, count = tc._abi.load(), len(ns)
    n_arr = (ctypes.c_int * count)(*ns)
    least = [r.clone() for r in rhos]
    work = torch.empty(int(lib.tc_batch_workspace_size(count, n_arr, tc.TC_FP64)) - 65536, dtype=torch.uint8, device="cuda")
    tc._abi.call("tc_batch_evolve", count, n_arr, (ctypes.c_void_p * count)(*[u.data_ptr() for u in Us]),
                 (ctypes.c_void_p * count)(*[r.data_ptr() for r in least]), steps, tc.TC_FP64, 0, None, None,
                 ctypes.c_void_p(work.data_ptr()), work.numel(),
                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    tc.sync_status()
    for n, a, b in zip(ns, outs, least):
        assert torch.equal(a, b) if n <= 6 else torch.max(torch.abs(a - b)).item() <= _bound(n, steps)

"""TC_FP64 on the tensor cores (residue products) against its DMMA form.

The DMMA form is reached by a workspace below what tc_workspace_size states.
Tolerance of one product, relative to the 2-norms of the two rows: each row
is rounded to half a unit of 2^-57.32 of its norm per entry, 2 K entries, so
2 sqrt(2 K) 2^-58.32 (Cauchy-Schwarz), plus 4 roundings of 2^-53 and, for the
DMMA sums, K 2^-52 (2 K additions in sequence of two products each).  A step
is two products with rows of U of norm 1 (unitary), and every entry's error
stays below that of the whole by the rows' norms.
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


def _bound(n, steps, scale=1.0):
    K = 1 << n
    return steps * 2 * scale * (2 * np.sqrt(2 * K) * 2.0 ** -58.32 + 4 * 2.0 ** -53 + K * 2.0 ** -52)


def _setup(tc, n, dt=0.1, seed=0):
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 70 + n + seed) * 5)), 1.013, 1.0)
    return p, tc.expm_model(p, dt)


def _dmma(tc, U, rho, n, steps, params, renorm=0):
    """tc_evolve(TC_FP64) in 64 KiB less than the tensor-core form's workspace."""
    out = rho.clone()
    obs = torch.empty((steps + 1, tc.obs_stride(n)), dtype=torch.float64, device="cuda")
    work = torch.empty(tc.workspace_size(n, tc.TC_FP64) - 65536, dtype=torch.uint8, device="cuda")
    p = params.c()
    tc._abi.call("tc_evolve", ctypes.c_void_p(U.data_ptr()), ctypes.c_void_p(out.data_ptr()), n, steps, tc.TC_FP64,
                 renorm, ctypes.byref(p), ctypes.c_void_p(obs.data_ptr()), ctypes.c_void_p(work.data_ptr()),
                 work.numel(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    tc.sync_status()
    return out, obs


@pytest.mark.parametrize("n,steps", [(7, 1), (7, 6), (8, 5), (9, 3), (10, 2), (11, 1)])
def test_tensor_core_form_equals_the_dmma_form(tc, n, steps):
    """n = 7 (one tile, single CTA), 8 .. 10 (pairs, one K chunk), 11 (two K chunks)."""
    p, U = _setup(tc, n)
    rho = torch.from_numpy(W.random_mixed_state(n, 3, 7 * n)[0]).cuda()
    a, oa = tc.evolve(U, rho, n, steps, "fp64", renorm_every=2, params=p)
    b, ob = _dmma(tc, U, rho, n, steps, p, renorm=2)
    assert not torch.equal(a, b)                       # two different routes
    assert torch.max(torch.abs(a - b)).item() < _bound(n, steps)
    assert torch.max(torch.abs(oa - ob)).item() < (1 << n) * _bound(n, steps)
    assert torch.equal(a, a.conj().T)


@pytest.mark.parametrize("n", [7, 9])
def test_any_rho_as_the_dmma_form_reads_it(tc, n):
    """The lower half of U rho U^dag, mirrored, for a rho that is not Hermitian; a large dt (U far from
    the identity)."""
    p, U = _setup(tc, n, dt=3.0)
    rng = np.random.default_rng(n)
    N = 1 << n
    rho = torch.from_numpy((rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))) / N).cuda()
    a, _ = tc.evolve(U, rho, n, 1, "fp64", params=p)
    b, _ = _dmma(tc, U, rho, n, 1, p)
    norm = torch.linalg.vector_norm(rho, dim=1).max().item()
    assert torch.max(torch.abs(a - b)).item() < _bound(n, 1, 4 * norm)
    same, _ = tc.evolve(U, rho, n, 0, "fp64", params=p)
    assert torch.equal(same, rho)


def test_rows_of_very_different_sizes(tc):
    """rho = S A S with S from 1 down to 2^-300: every row keeps the accuracy of its own norm in
    X = U rho; rho' mixes the rows, so its bound is the largest row's."""
    n = 8
    N = 1 << n
    p, U = _setup(tc, n)
    rng = np.random.default_rng(1)
    A = rng.standard_normal((N, 5)) + 1j * rng.standard_normal((N, 5))
    s = 2.0 ** -np.linspace(0, 300, N)
    M = s[:, None] * (A @ A.conj().T) * s[None, :] / 5
    rho = torch.from_numpy(M / np.trace(M).real).cuda()
    eye = torch.eye(N, dtype=torch.complex128, device="cuda")
    a, _ = tc.evolve(U, rho, n, 2, "fp64", params=p)
    b, _ = _dmma(tc, U, rho, n, 2, p)
    assert torch.max(torch.abs(a - b)).item() < _bound(n, 2)
    # with U = 1 the product is rho itself, entry by entry (the diagonal is kept in FP64)
    c, _ = tc.evolve(eye, rho, n, 1, "fp64", params=p)
    low = torch.tril(rho)
    assert torch.equal(torch.tril(c, -1), torch.tril(low, -1))


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_entries_spread_as_in_the_dmma_form(tc, bad):
    n = 7
    p, U = _setup(tc, n)
    rho = torch.from_numpy(W.random_mixed_state(n, 2, 5)[0]).cuda()
    rho[3, 5] = bad
    a, _ = tc.evolve(U, rho, n, 1, "fp64", params=p)
    out = rho.clone()
    b, _ = _dmma(tc, U, out, n, 1, p)
    # nothing finite is left but the diagonal's imaginary part, which both forms write as 0
    assert torch.equal(torch.isfinite(torch.view_as_real(a)), torch.isfinite(torch.view_as_real(b)))
    assert not torch.isfinite(a.real).any()


def test_gradient_on_the_tensor_cores_with_squarings(tc, oracle):
    """A large dt makes the Frechet recurrence square (D <- X D + D X); against the oracle's tangent."""
    n, dt, steps = 7, 2.0, 3
    g = W.draw_couplings(n, 4) * 20
    p = tc.Params(n, list(map(float, g)), 1.05, 1.0)
    U = tc.expm_model(p, dt)
    N = 1 << n
    rho0 = torch.zeros((N, N), dtype=torch.complex128, device="cuda")
    rho0[-1, -1] = 1.0
    O = ((torch.arange(N, device="cuda") >> (n - 2)) & 1).to(torch.float64)
    grad, loss = tc.evolve_backward(p, dt, steps, rho0, U, O, ckpt_every=2)
    grad2, loss2 = tc.evolve_backward(p, dt, steps, rho0, U, O, ckpt_every=2, precision="ozaki")
    assert torch.equal(grad, grad2) and loss == loss2   # one route for both from n = 7 on
    # the DMMA form (its planes: 11 + 2 checkpoints + 2 states of two N x N matrices, one real one, the small buffers)
    cm = 2 * 8 * N * N
    for size, tol in ((15 * cm + cm // 2 + 16384, 1e-11),):
        work = torch.empty(size, dtype=torch.uint8, device="cuda")
        ref = (ctypes.c_double * (n + 2))()
        c = p.c()
        tc._abi.call("tc_evolve_backward", ctypes.byref(c), dt, steps, ctypes.c_void_p(rho0.data_ptr()),
                     ctypes.c_void_p(U.data_ptr()), 2, tc.TC_FP64, ctypes.c_void_p(O.data_ptr()), ref, None,
                     ctypes.c_void_p(work.data_ptr()), work.numel(),
                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        ref = torch.tensor(list(ref), dtype=torch.float64)
        assert torch.max(torch.abs(grad - ref)).item() <= tol * torch.max(torch.abs(ref)).item()


@pytest.mark.parametrize("n,degree,squarings", [(8, 0, -1), (8, 6, 3), (9, 0, -1), (11, 12, 1)])
def test_expm_on_the_tensor_cores_equals_the_dmma_form(tc, n, degree, squarings):
    """One tile (n = 8), one and two K chunks; plans with and without squarings.  Every entry of the
    polynomials is bounded by 1 (cos, sin of B), each product within 2 sqrt(K) 2^-58.32 of its rows'
    norms (<= 1) plus roundings, the DMMA sums K 2^-53; at most 8 + 3 squarings products, doubled per
    squaring."""
    N = 1 << n
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 5) * 4)), 1.01, 1.0)
    H = tc.build_hamiltonian(p)
    a = tc.expm(H, n, 0.3, taylor_degree=degree, squarings=squarings)
    b = torch.empty_like(a)
    # one scratch matrix and a bit less than the tensor-core form needs
    work = torch.empty(tc.workspace_size(n, tc.TC_FP64, tc.TC_OP_EXPM) - 8 * N * N - 65536, dtype=torch.uint8,
                       device="cuda")
    opts = tc._abi.tc_expm_opts(degree, squarings, 1)
    tc._abi.call("tc_expm", ctypes.c_void_p(H.data_ptr()), n, 0.3, ctypes.byref(opts), ctypes.c_void_p(b.data_ptr()),
                 ctypes.c_void_p(work.data_ptr()), work.numel(),
                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    one = 2 * np.sqrt(N) * 2.0 ** -58.32 + 4 * 2.0 ** -53 + N * 2.0 ** -53
    assert torch.max(torch.abs(a - b)).item() < 2 ** max(squarings, 0) * (8 + 3 * max(squarings, 0)) * one
    assert not torch.equal(a, b)
    assert torch.equal(a, a.T)

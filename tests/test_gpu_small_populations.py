"""Small populations and coherences in TC_FP64 on the tensor cores: relative to themselves, not to the matrix.

U falls by a factor g dt for every atom that differs, and a state a few steps from a basis state spans as many
orders as the GPU's FP64 form has to carry.  References are numpy's from the same U.

Tolerances.  A product's error at (i, j) is below K 2^-55 a_i sqrt(rho_jj), a_i^2 = sum_k |U_ik|^2 rho_kk (the
operands' half units, 2 sqrt(2 K) 2^-58.32 of their rows' norms after the column scales, rows of up to
2 sqrt(K rho_jj)), plus 8 roundings; the second product's at most K 2^-55 a_i sqrt(rho'_jj).  For a pure state
with q = |U| |psi| both stay below q_i q_j, and numpy's sums of K terms are within K 2^-53 of it.  Each product
after an error passes it on once (q of q).  So a step is within 2 (K 2^-55 + K 2^-53 + 8 2^-53) q_i q_j.
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


def _tol(K, steps):
    return steps * 2 * (K * 2.0 ** -55 + K * 2.0 ** -53 + 8 * 2.0 ** -53)


def _setup(tc, n, dt=0.05):
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 3))), 1.002, 1.0)
    return p, tc.expm_model(p, dt)


def _pure(U, psi, steps):
    q = np.abs(psi)
    for _ in range(steps):
        q = np.abs(U) @ q
        psi = U @ psi
    return psi, q


def _check(rho, psi, q, steps):
    """Entry by entry; where U's Taylor series stops short of an entry, q and so rho are exactly zero."""
    err, scale = np.abs(rho.cpu().numpy() - np.outer(psi, psi.conj())), np.outer(q, q)
    assert (err <= _tol(len(psi), steps) * scale).all(), (err[scale > 0] / scale[scale > 0]).max()


@pytest.mark.parametrize("n,steps,start", [(7, 1, -1), (8, 1, -1), (8, 7, -1), (8, 40, 0x5A), (9, 3, 0), (10, 2, -1),
                                           (11, 1, -1)])
def test_every_entry_of_a_state_near_a_basis_state(tc, n, steps, start):
    """One tile, one and two K chunks; direct reads and writes of rho and steps in graphs."""
    p, U = _setup(tc, n)
    N = 1 << n
    psi = np.zeros(N, np.complex128)
    psi[start] = 1.0
    rho0 = torch.from_numpy(np.outer(psi, psi.conj())).cuda()
    rho, obs = tc.evolve(U, rho0, n, steps, "fp64", params=p)
    psi, q = _pure(U.cpu().numpy(), psi, steps)
    _check(rho, psi, q, steps)
    pop = np.array([bin(s).count("1") for s in range(N)])
    for m in range(n + 1):   # P(m); the row's sums add at most N roundings
        want, scale = (np.abs(psi) ** 2)[pop == n - m].sum(), (q ** 2)[pop == n - m].sum()
        assert abs(obs[-1, n + 1 + m].item() - want) <= (_tol(N, steps) + N * 2.0 ** -53) * scale, m


def test_small_populations_in_a_batch_and_from_host_memory(tc):
    ns, steps = [8, 7, 9], 3
    ps, Us = zip(*[_setup(tc, n) for n in ns])
    rhos = [torch.from_numpy(W.all_excited_rho(n)).cuda() for n in ns]
    outs, _ = tc.batch_evolve(list(Us), rhos, steps, "fp64", params=list(ps))
    for n, U, out in zip(ns, Us, outs):
        psi, q = _pure(U.cpu().numpy(), W.all_excited_state(n), steps)
        _check(out, psi, q, steps)
    host = torch.from_numpy(W.all_excited_rho(8))
    tc.evolve_host(Us[0], host, 8, steps, "fp64", params=ps[0])
    assert torch.equal(host, outs[0].cpu())


def test_incoherent_state_with_weights_of_every_size(tc):
    """rho diagonal, 1 down to 2^-200 in an order of its own: P_i = sum_k |U_ik|^2 w_k has no cancellation."""
    n = 8
    N = 1 << n
    p, U = _setup(tc, n)
    w = 2.0 ** -np.linspace(0, 200, N)[np.random.default_rng(2).permutation(N)]
    rho, _ = tc.evolve(U, torch.from_numpy(np.diag(w).astype(np.complex128)).cuda(), n, 1, "fp64", params=p)
    want = (np.abs(U.cpu().numpy()) ** 2) @ w
    got = np.diagonal(rho.cpu().numpy()).real
    # a_i^2 = P_i and sqrt(rho'_ii) = a_i here; the first product's errors add up over k: sqrt(K) of them at most
    assert (np.abs(got - want) / want).max() < np.sqrt(N) * _tol(N, 1)


def test_matrices_that_are_no_states(tc):
    """A zero diagonal with large and small entries off it, a zero row and column, one empty row only: errors
    relative to the largest entry, against numpy (K 2^-53 of sums of K products of entries up to 1, twice; after the
    column scales operands' entries stay below twice the root of the largest entry, hence 16 times the half units)."""
    n = 8
    N = 1 << n
    p, U = _setup(tc, n, dt=2.0)
    rng = np.random.default_rng(4)
    A = (rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))) * 2.0 ** -rng.integers(0, 60, (N, N))
    A = A + A.conj().T
    np.fill_diagonal(A, 0.0)
    A[5], A[:, 5] = 0.0, 0.0
    B = A.copy()
    B[9] = 0.0   # not Hermitian: the lower half of U rho U^H
    u = U.cpu().numpy()
    bound = 2 * N * (16 * 2.0 ** -55 + 2.0 ** -52) * np.abs(A).max() * np.sqrt(N)
    for M in (A, B):
        rho, _ = tc.evolve(U, torch.from_numpy(M.copy()).cuda(), n, 1, "fp64", params=p)
        want = np.tril(u @ M @ u.conj().T)
        assert np.abs(np.tril(rho.cpu().numpy()) - want)[np.tril_indices(N, -1)].max() < bound


def test_small_populations_of_the_open_system(tc):
    """Blocks on the tensor cores against the same blocks on the DMMA (a smaller workspace), entry by entry on the
    diagonal: without interference (g t << 1) the sums of magnitudes are within twice the populations."""
    n, steps, kappa, dt = 10, 3, 0.02, 0.05
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 3))), 1.002, 1.0)
    lay = tc.lindblad_layout(n)
    U = tc.lindblad_propagators(p, dt)
    rho = torch.zeros(lay.total, dtype=torch.complex128, device="cuda")
    rho[-1] = 1.0
    a, _ = tc.lindblad_evolve(p, kappa, dt, U, rho, steps, "fp64")
    b = rho.clone()
    work = torch.empty(tc.workspace_size(n, tc.TC_FP64, tc._abi.TC_OP_LINDBLAD) - 65536, dtype=torch.uint8, device="cuda")
    c = p.c()
    tc._abi.call("tc_lindblad_evolve", ctypes.byref(c), kappa, dt, ctypes.c_void_p(U.data_ptr()),
                 ctypes.c_void_p(b.data_ptr()), steps, tc.TC_FP64, 0, None, ctypes.c_void_p(work.data_ptr()),
                 work.numel(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    tc.sync_status()
    for k, (x, y) in enumerate(zip(lay.blocks(a), lay.blocks(b))):
        x, y = x.diagonal().real, y.diagonal().real
        big = y > 1e-280
        assert ((x - y).abs()[big] / y[big]).max().item() < 4 * np.sqrt(1 << n) * _tol(1 << n, steps) if big.any() else True, k


@pytest.mark.parametrize("n", [8, 10, 11])
def test_small_entries_of_the_exponential(tc, n):
    """tc_expm on the tensor cores against the DMMA, the same polynomial: with both diagonals apart a product's error
    is relative to the off-diagonal parts of its rows, beta for B = (H - mu) dt, beta^2 and more for every matrix of
    the polynomial, so below beta^4 in all; the DMMA sums' N roundings of sums like the entry itself."""
    N, dt = 1 << n, 0.05
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 3))), 1.002, 1.0)
    H = tc.build_hamiltonian(p)
    a, b = tc.expm(H, n, dt), tc.expm(H, n, dt, precision="fp64_dmma")
    beta = (torch.linalg.vector_norm(H - torch.diag(H.diagonal()), dim=1).max() * dt).item()
    assert ((a - b).abs() <= N * 2.0 ** -52 * (b.abs() + beta ** 4)).all()


@pytest.mark.parametrize("n,steps,ckpt", [(8, 2, 2), (8, 20, 6), (7, 3, 1)])
def test_gradient_of_a_small_loss(tc, n, steps, ckpt):
    """L = P(m photons) from the all-excited state, down to 1e-33, against the DMMA form of the same series: 4 products
    a step, three a Taylor term (at most 20), each within K 2^-52 of its sum of magnitudes."""
    N, dt = 1 << n, 0.05
    p, U = _setup(tc, n, dt)
    rho = torch.from_numpy(W.all_excited_rho(n)).cuda()
    pop = np.array([bin(s).count("1") for s in range(N)])
    for m in (1, 2, 4, 6):
        O = torch.from_numpy((pop == n - m).astype(np.float64)).cuda()
        a, la = tc.evolve_backward(p, dt, steps, rho, U, O, ckpt_every=ckpt)
        b, lb = tc.evolve_backward(p, dt, steps, rho, U, O, ckpt_every=ckpt, precision="fp64_dmma")
        tol = (4 * steps + 60) * N * 2.0 ** -52
        assert abs(la - lb) <= tol * lb, m
        assert (a - b).abs().max().item() <= tol * b.abs().max().item(), m

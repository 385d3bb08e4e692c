"""The work a user of this framework has it do, case by case: the step loop in every precision, from host memory too,
batches of uneven systems, the open system, the gradient, and the propagator.

Every case goes through the torch-facing entry points of ``paper_2403_06937_gb300``.  The parameters are those of the
workloads in ``workloads.py``: couplings uniform in [0.005, 0.015), omega_a = 1.002, omega_c = 1, dt = 0.05.

``exact`` uses none of the framework: it applies the Hamiltonian of Eq. 4 to state vectors as n index permutations and
sums the Taylor series of e^{-iH dt} to convergence in complex128, so rho = sum_r w_r psi_r psi_r^dag costs one thin
product at any n.
"""
import math

import numpy as np
import torch

import paper_2403_06937_gb300 as tc

OMEGA_A, OMEGA_C, DT, KAPPA = 1.002, 1.0, 0.05, 0.02
PRECISIONS = ("fp64", "bf16x3", "tf32", "tf32x3", "ozaki")


def listed():
    return [
        # A program that drives the smallest systems itself, one step per call, and looks at rho in between.
        dict(name="step_n7_fp64", kind="evolve", n=7, steps=1, precision="fp64", start="mixed", renorm=0),
        # The plain method: 100 steps at n = 8 from the all-excited state, one observable row per step.
        dict(name="run_n8_fp64", kind="evolve", n=8, steps=100, precision="fp64", start="excited", renorm=0),
        # A middle size in the precision form, renormalised as in the n = 14 workload: launches and tails count.
        dict(name="run_n10_bf16x3", kind="evolve", n=10, steps=50, precision="bf16x3", start="mixed", renorm=50),
        # FP64-accurate products on the tensor cores, at the gradient workload's size.
        dict(name="run_n11_ozaki", kind="evolve", n=11, steps=8, precision="ozaki", start="mixed", renorm=0),
        # The plain method at scale: a step of the n = 12 workload.
        dict(name="step_n12_fp64", kind="evolve", n=12, steps=1, precision="fp64", start="mixed", renorm=0),
        # Split TF32, between the sizes that the other cases have.
        dict(name="run_n13_tf32x3", kind="evolve", n=13, steps=4, precision="tf32x3", start="mixed", renorm=0),
        # The precision form at full size: the n = 14 workload in its dense phase.
        dict(name="run_n14_bf16x3", kind="evolve", n=14, steps=3, precision="bf16x3", start="mixed", renorm=0),
        # The state lives in page-locked host memory and goes in and out with each call.
        dict(name="host_n13_bf16x3", kind="host", n=13, steps=2, precision="bf16x3", start="mixed", renorm=0),
        # Many systems of uneven size in one call, sizes drawn as in the batch workload.
        dict(name="batch32_bf16x3", kind="batch", count=32, n_lo=6, n_hi=12, sizes=2, steps=10, precision="bf16x3",
             start="mixed", renorm=0),
        # The open system: ragged excitation blocks, the damping channel and the block products.
        dict(name="open_n11_bf16x3", kind="open", n=11, steps=4, precision="bf16x3", start="excited", renorm=50),
        # One gradient of the loss of the gradient workload: forward and backward through the autograd function.
        dict(name="grad_n8_fp64", kind="grad", n=8, steps=100, precision="fp64", start="mixed", ckpt=20),
        # Set-up by the paper's own route: dense H, then its exponential.
        dict(name="expm_n11", kind="expm", n=11, shift=True),
    ]


# Seconds that one step of 8 N^3 + 4 N^3 FLOPs may be taken to last in each precision; keeps a drawn case below the
# largest listed one.
_RATE = {"fp64": 1.0e12, "bf16x3": 2.5e14, "tf32": 6.0e14, "tf32x3": 2.5e14, "ozaki": 2.5e13}


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _most_steps(n, precision, seconds=0.35, factor=1.0, most=200):
    per = max(2.0e-3 if precision == "ozaki" else 2.0e-4, factor * 12.0 * 8.0 ** n / _RATE[precision])
    return max(1, min(most, int(seconds / per)))


def draw(rng):
    kind = rng.choice(["evolve"] * 5 + ["host", "batch", "batch", "open", "open", "grad", "expm", "model"])
    start = rng.choice(["mixed", "excited"])
    precision = rng.choice(PRECISIONS)
    if kind == "evolve":
        n = rng.randint(7 if precision == "ozaki" else 6, {"fp64": 11, "ozaki": 13}.get(precision, 14))
        return dict(kind=kind, n=n, steps=_log_int(rng, 1, _most_steps(n, precision)), precision=precision, start=start,
                    renorm=rng.choice([0, 0, rng.randint(1, 50)]))
    if kind == "host":
        precision = rng.choice(["bf16x3", "tf32x3", "fp64", "ozaki"])
        n = rng.randint(7, {"fp64": 10, "ozaki": 12}.get(precision, 13))
        return dict(kind=kind, n=n, steps=_log_int(rng, 1, _most_steps(n, precision, 0.15, most=10)), precision=precision,
                    start=start, renorm=0)
    if kind == "batch":
        n_hi = rng.randint(8, {"fp64": 9, "ozaki": 11}.get(precision, 12))
        count = _log_int(rng, 2, 32)
        return dict(kind=kind, count=count, n_lo=7 if precision == "ozaki" else 6, n_hi=n_hi, sizes=rng.randrange(1 << 20),
                    steps=_log_int(rng, 1, _most_steps(n_hi, precision, 0.3, factor=max(1.0, count / 3), most=50)),
                    precision=precision, start=start, renorm=0)
    if kind == "open":
        n = rng.randint(7, {"fp64": 9, "ozaki": 10}.get(precision, 12))
        return dict(kind=kind, n=n, steps=_log_int(rng, 1, _most_steps(n, precision, 0.2, factor=4.0, most=20)),
                    precision=precision, start="excited", renorm=rng.choice([0, rng.randint(1, 10)]))
    if kind == "grad":
        precision = rng.choice(["fp64", "ozaki"])
        n = rng.randint(7, 9 if precision == "fp64" else 10)
        steps = _log_int(rng, 2, _most_steps(n, precision, 0.2, factor=4.0, most=60))
        # after so few steps from the all-excited state the frequency gradients are rounding noise
        return dict(kind=kind, n=n, steps=steps, precision=precision, start="mixed", ckpt=rng.randint(1, steps))
    if kind == "expm":
        return dict(kind=kind, n=rng.randint(6, 11), shift=rng.random() < 0.7)
    return dict(kind=kind, n=rng.randint(6, 13), shift=rng.random() < 0.7)


# ------------------------------------------------------------------ inputs, from the seed alone


def _sizes(case):
    """The n of every system: the case's systems, or the one that it names."""
    if case["kind"] != "batch":
        return [case["n"]]
    return [int(n) for n in np.random.default_rng(case["sizes"]).integers(case["n_lo"], case["n_hi"] + 1, size=case["count"])]


def _couplings(case, seed):
    rng = np.random.default_rng([seed, 1])
    return [rng.uniform(0.005, 0.015, size=n) for n in _sizes(case)]


def _states(case, seed, device="cuda"):
    """Per system, (psi, w): rho = sum_r w_r psi[:, r] psi[:, r]^dag."""
    gen = torch.Generator(device=device).manual_seed(seed)
    out = []
    for n in _sizes(case):
        N = 1 << n
        if case["start"] == "excited":
            psi = torch.zeros((N, 1), dtype=torch.complex128, device=device)
            psi[-1] = 1.0
            w = torch.ones(1, dtype=torch.float64, device=device)
        else:
            psi = torch.randn((N, 4), dtype=torch.complex128, device=device, generator=gen)
            psi = psi / torch.linalg.vector_norm(psi, dim=0)
            w = torch.rand(4, dtype=torch.float64, device=device, generator=gen) + 0.1
            w = w / w.sum()
        out.append((psi, w))
    return out


def _rho(psi, w):
    rho = (psi * w) @ psi.mH
    return (rho + rho.mH) / 2


def _observable(n, seed, device="cuda"):
    """A diagonal observable: the excited population of one atom, drawn from the seed."""
    atom = int(np.random.default_rng([seed, 2]).integers(1, n + 1))
    return ((torch.arange(1 << n, device=device) >> (n - atom)) & 1).to(torch.float64)


def _params(case, seed):
    return [tc.Params(len(g), [float(x) for x in g], OMEGA_A, OMEGA_C) for g in _couplings(case, seed)]


def prepare(case, seed):
    kind, params = case["kind"], _params(case, seed)
    p = params[0]
    state = dict(case=case, p=p)
    if kind in ("expm", "model"):
        return state
    if kind == "open":
        lay = tc.lindblad_layout(p.n)
        rho = torch.zeros(lay.total, dtype=torch.complex128, device="cuda")
        rho[-1] = 1.0  # the top block's last basis string: all atoms excited, no photon
        return state | dict(U=tc.lindblad_propagators(p, DT), rho=rho)
    rhos = [_rho(psi, w) for psi, w in _states(case, seed)]
    if kind == "grad":
        return state | dict(g=torch.tensor(list(p.g), dtype=torch.float64, requires_grad=True),
                            wa=torch.tensor(OMEGA_A, dtype=torch.float64, requires_grad=True),
                            wc=torch.tensor(OMEGA_C, dtype=torch.float64, requires_grad=True),
                            rho=rhos[0], O=_observable(p.n, seed))
    if kind == "batch":
        return state | dict(Us=[tc.expm_model(q, DT) for q in params], rhos=rhos, params=params)
    state["U"] = tc.expm_model(p, DT)
    if kind == "host":
        rho = torch.empty(rhos[0].shape, dtype=torch.complex128, pin_memory=True)
        rho.copy_(rhos[0])
        obs = torch.empty((case["steps"] + 1, tc.obs_stride(p.n)), dtype=torch.float64, pin_memory=True)
        return state | dict(rho=rho, obs=obs)
    return state | dict(rho=rhos[0])


def run(state):
    case, p = state["case"], state["p"]
    kind = case["kind"]
    if kind == "expm":
        return tc.expm(tc.build_hamiltonian(p), p.n, DT, shift=case["shift"])
    if kind == "model":
        return tc.expm_model(p, DT, shift=case["shift"])
    if kind == "grad":
        loss = tc.EvolveFn.apply(state["g"], state["wa"], state["wc"], state["rho"], state["O"], DT, case["steps"],
                                 case["ckpt"], tc.TC_COUPLING_BOSONIC, case["precision"])
        return (loss.detach(),) + torch.autograd.grad(loss, (state["g"], state["wa"], state["wc"]))
    if kind == "open":
        return tc.lindblad_evolve(p, KAPPA, DT, state["U"], state["rho"], case["steps"], case["precision"],
                                  renorm_every=case["renorm"])
    if kind == "batch":
        return tc.batch_evolve(state["Us"], state["rhos"], case["steps"], case["precision"],
                               renorm_every=case["renorm"], params=state["params"])
    if kind == "host":
        tc.evolve_host(state["U"], state["rho"], p.n, case["steps"], case["precision"], renorm_every=case["renorm"],
                       params=p, obs_host=state["obs"])
        return state["rho"], state["obs"]
    return tc.evolve(state["U"], state["rho"], p.n, case["steps"], case["precision"], renorm_every=case["renorm"],
                     params=p)


# ------------------------------------------------------------------ what one pass cannot do without


def _block_dims(n):
    return [sum(math.comb(n, j) for j in range(k + 1)) for k in range(n + 1)]


def work(case):
    kind = case["kind"]
    if kind in ("expm", "model"):
        # the route through the dense H reads it once; the result is written once; one Taylor product at least
        N = 1 << case["n"]
        dense = kind == "expm"
        return {"bytes": (24.0 if dense else 16.0) * N * N, "flops": 8.0 * N ** 3 if dense else 8.0 * case["n"] * N * N}
    # U and rho read once, rho' written once; per step X = U rho (8 d^3) and the Hermitian half of X U^dag (4 d^3)
    dims = _block_dims(case["n"]) if kind == "open" else [1 << n for n in _sizes(case)]
    flops = 12.0 * case["steps"] * sum(float(d) ** 3 for d in dims)
    if kind == "grad":
        # forward and adjoint steps and the accumulation of rho_k Lambda_k; only rho_0 is read
        return {"bytes": 16.0 * dims[0] ** 2, "flops": flops * 2 + 8.0 * case["steps"] * float(dims[0]) ** 3}
    return {"bytes": 48.0 * sum(float(d) ** 2 for d in dims), "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits, by another route


class _Model:
    """H of Eq. 4 on columns of a matrix, as n index permutations: no dense matrix is formed."""

    def __init__(self, n, g, wa, wc, device="cuda"):
        s = torch.arange(1 << n, device=device)
        pop = sum((s >> b) & 1 for b in range(n))
        self.n, self.pop, self.g = n, pop, g
        self.diag = wc * (n - pop).to(torch.float64) + wa * pop.to(torch.float64)
        self.flip = [s ^ (1 << (n - 1 - i)) for i in range(n)]
        # photons of the excited-side string: one fewer than those of the string with the atom relaxed
        self.root = [torch.sqrt((n - pop + ((s >> (n - 1 - i)) & 1)).to(torch.float64)) for i in range(n)]

    def apply(self, x):
        y = self.diag[:, None] * x
        for i in range(self.n):
            y = y + (self.g[i] * self.root[i])[:, None] * x[self.flip[i]]
        return y

    def propagate(self, x, dt, shift):
        """e^{-i (H - shift) dt} x."""
        term, total = x, x
        for k in range(1, 60):
            term = (self.apply(term) - shift * term) * (-1j * dt / k)
            total = total + term
            if float(term.detach().abs().max()) < 1e-19:
                break
        return total

    def row(self, psi, w):
        """One observable row of sum_r w_r psi_r psi_r^dag."""
        n, prob = self.n, (psi.abs() ** 2) @ w
        p_i = [prob[((torch.arange(1 << n, device=psi.device) >> (n - 1 - i)) & 1) == 1].sum() for i in range(n)]
        p_m = [prob[self.pop == n - m].sum() for m in range(n + 1)]
        gram = psi.mH @ psi
        energy = ((psi.conj() * self.apply(psi)).real.sum(0) * w).sum()
        purity = ((gram.abs() ** 2) * w[:, None] * w[None, :]).sum()
        return torch.stack(p_i + [(prob * (n - self.pop)).sum()] + p_m + [prob.sum(), purity, energy])


def _exact_system(g, psi, w, steps):
    m = _Model(len(g), [float(x) for x in g], OMEGA_A, OMEGA_C)
    shift = float(m.diag.mean())
    rows = [m.row(psi, w)]
    for _ in range(steps):
        psi = m.propagate(psi, DT, shift)
        rows.append(m.row(psi, w))
    return (psi * w) @ psi.mH, torch.stack(rows)


def _exact_open(case, g):
    """The split step on the excitation blocks, densely."""
    n, steps = case["n"], case["steps"]
    eta = math.exp(-KAPPA * DT / 2)
    m = _Model(n, [float(x) for x in g], OMEGA_A, OMEGA_C)
    s = torch.arange(1 << n, device="cuda")
    order = torch.argsort(m.pop * (1 << n) + s)
    dims = _block_dims(n)
    where = torch.empty_like(order)
    where[order] = s
    hams, props, photons = [], [], []
    for k, d in enumerate(dims):
        b = order[:d]
        ph = k - m.pop[b]
        h = torch.diag(OMEGA_C * ph.double() + OMEGA_A * m.pop[b].double())
        for i in range(n):
            to = where[b ^ (1 << (n - 1 - i))]
            at = torch.nonzero(((b >> (n - 1 - i)) & 1) == 1)[:, 0]  # excited strings: the partner has one photon more
            v = float(g[i]) * torch.sqrt((ph[at] + 1).double())
            h[to[at], at] = v
            h[at, to[at]] = v
        shift = float(h.diagonal().mean())
        x = ((h - shift * torch.eye(d, dtype=h.dtype, device=h.device)) * DT).to(torch.complex128)
        u = term = torch.eye(d, dtype=torch.complex128, device="cuda")
        for j in range(1, 40):
            term = (x @ term) * (-1j / j)
            u = u + term
            if float(term.abs().max()) < 1e-19:
                break
        hams.append(h)
        props.append(u)
        photons.append(ph)
    rho = [torch.zeros((d, d), dtype=torch.complex128, device="cuda") for d in dims]
    rho[n][-1, -1] = 1.0

    def damp(rho):
        out = []
        for k, d in enumerate(dims):
            acc = torch.zeros_like(rho[k])
            for j in range(n - k + 1):
                # Kraus operator j takes q + j photons (block k + j) to q: sqrt(C(q+j, j) (1-eta)^j eta^q)
                q = photons[k]
                f = torch.tensor([math.sqrt(math.comb(int(v) + j, j) * (1 - eta) ** j * eta ** int(v)) for v in range(n + 1)],
                                 dtype=torch.float64, device="cuda")[q]
                acc += f[:, None] * f[None, :] * rho[k + j][:d, :d]
            out.append(acc)
        return out

    def row(rho):
        prob = torch.zeros(1 << n, dtype=torch.float64, device="cuda")
        p_m = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
        purity = energy = mean = 0.0
        for k, d in enumerate(dims):
            diag = rho[k].diagonal().real
            prob[order[:d]] += diag
            p_m.index_add_(0, photons[k], diag)
            mean = mean + (diag * photons[k]).sum()
            purity = purity + (rho[k].abs() ** 2).sum()
            energy = energy + (hams[k] * rho[k].real.mT).sum()
        p_i = torch.stack([prob[((s >> (n - 1 - i)) & 1) == 1].sum() for i in range(n)])
        return torch.cat([p_i, torch.stack([mean]), p_m, torch.stack([prob.sum(), purity, energy])])

    rows = [row(rho)]
    for t in range(steps):
        rho = damp(rho)
        rho = [u @ r @ u.mH for u, r in zip(props, rho)]
        rho = damp(rho)
        if case["renorm"] and (t + 1) % case["renorm"] == 0:
            trace = sum(r.diagonal().real.sum() for r in rho)
            rho = [r / trace for r in rho]
        rows.append(row(rho))
    return torch.cat([r.reshape(-1) for r in rho]), torch.stack(rows)


def exact(case, seed):
    kind, gs = case["kind"], _couplings(case, seed)
    if kind in ("expm", "model"):
        m = _Model(case["n"], [float(x) for x in gs[0]], OMEGA_A, OMEGA_C)
        shift = float(m.diag.mean())
        one = torch.eye(1 << case["n"], dtype=torch.complex128, device="cuda")
        return m.propagate(one, DT, shift) * complex(math.cos(shift * DT), -math.sin(shift * DT))
    if kind == "open":
        return _exact_open(case, gs[0]) if case["n"] <= 11 else None
    states = _states(case, seed)
    if kind == "grad":
        psi, w = states[0]
        g = torch.tensor(gs[0], dtype=torch.float64, requires_grad=True)
        wa = torch.tensor(OMEGA_A, dtype=torch.float64, requires_grad=True)
        wc = torch.tensor(OMEGA_C, dtype=torch.float64, requires_grad=True)
        m = _Model(case["n"], g.cuda(), wa.cuda(), wc.cuda())
        shift = float(m.diag.detach().mean())
        for _ in range(case["steps"]):
            psi = m.propagate(psi, DT, shift)
        loss = (((psi.abs() ** 2) @ w) * _observable(case["n"], seed)).sum()
        return (loss.detach(),) + torch.autograd.grad(loss, (g, wa, wc))
    got = [_exact_system(g, psi, w, case["steps"]) for g, (psi, w) in zip(gs, states)]
    if kind == "batch":
        return [r for r, _ in got], [o for _, o in got]
    return got[0]

"""The step loops on the library's own streams: repeated graphs, and callers on several threads.

All comparisons are bitwise: the same launches on the same operands, only
enqueued differently (captured steps against plain launches, which timing
selects), or by another thread.
"""
import threading

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


def _setup(tc, n, seed=0):
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 50 + n + seed) * 5)), 1.013, 1.0)
    rho = torch.from_numpy(W.random_mixed_state(n, 2, 3 * n + seed)[0]).cuda()
    return p, tc.expm_model(p, 0.1), rho


# one graph; growing ones; the graph of 64 steps again (56 = 8 + 16 + 32 before it), with renormalisation in no
# step, between the graphs of 64, and at several places in each
@pytest.mark.parametrize("n,precision,steps,renorm", [
    (7, "fp64", 9, 0), (7, "fp64", 26, 0), (7, "fp64", 185, 0), (7, "fp64", 186, 0), (7, "fp64", 330, 150),
    (7, "fp64", 250, 64), (7, "fp64", 250, 17), (7, "fp64", 200, 1), (5, "fp64", 260, 65), (5, "fp64", 190, 3),
    (8, "bf16x3", 185, 0), (8, "bf16x3", 190, 25), (6, "tf32", 200, 7)])
def test_repeated_steps_equal_plain_launches(tc, n, precision, steps, renorm):
    p, U, rho = _setup(tc, n)
    a, oa = tc.evolve(U, rho, n, steps, precision, renorm_every=renorm, params=p)
    c, _ = tc.evolve(U, rho, n, steps, precision, renorm_every=renorm, params=p, observe=False)
    try:
        tc.timing_enable(True)
        b, ob = tc.evolve(U, rho, n, steps, precision, renorm_every=renorm, params=p)
    finally:
        tc.timing_enable(False)
    tc.sync_status()
    assert torch.equal(a, b) and torch.equal(oa, ob) and torch.equal(a, c)


def test_callers_on_several_threads(tc):
    """Runs, batches and gradients from six threads at once, each on a stream of its own."""
    p, U, rho = _setup(tc, 7)
    O = torch.arange(128, dtype=torch.float64, device="cuda") / 128

    def work(i):
        if i % 3 == 0:
            return list(tc.evolve(U, rho, 7, 40, "fp64", params=p))
        if i % 3 == 1:
            outs, obs = tc.batch_evolve([U, U], [rho, rho], 3, "fp64", params=[p, p])
            return outs + obs
        grad, loss = tc.evolve_backward(p, 0.1, 12, rho, U, O, ckpt_every=4)
        return [grad, torch.tensor([loss], dtype=torch.float64)]

    want = [[x.clone() for x in work(i)] for i in range(3)]
    torch.cuda.synchronize()
    bad = []

    def run(i):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(6):
                got = work(i)
                s.synchronize()
                if not all(torch.equal(x, y) for x, y in zip(got, want[i % 3])):
                    bad.append(i)

    ts = [threading.Thread(target=run, args=(i,)) for i in range(6)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    tc.sync_status()
    assert not bad

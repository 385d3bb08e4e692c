"""The stream sets that the library keeps between calls: few, and given back on request."""
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


def test_idle_stream_sets_are_bounded_and_given_back(tc):
    n, steps = 6, 12
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 1))), 1.002, 1.0)
    U = tc.expm_model(p, 0.1)
    rho = torch.from_numpy(W.random_mixed_state(n, 2, 1)[0]).cuda()
    want, _ = tc.evolve(U, rho, n, steps, "fp64", params=p)
    torch.cuda.synchronize()
    got, gate = {}, threading.Barrier(5)

    def run(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            gate.wait()
            for _ in range(4):
                got[i] = tc.evolve(U, rho, n, steps, "fp64", params=p)[0]
            torch.cuda.current_stream().synchronize()

    ts = [threading.Thread(target=run, args=(i,)) for i in range(5)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    outs, _ = tc.batch_evolve([U, U, U], [rho] * 3, steps, "fp64", params=[p] * 3)
    # given back while the batch may still run: its work completes
    assert 1 <= tc.release_idle() <= 2
    assert tc.release_idle() == 0
    again, _ = tc.evolve(U, rho, n, steps, "fp64", params=p)
    torch.cuda.synchronize()
    tc.sync_status()
    for x in list(got.values()) + outs + [again]:
        assert torch.equal(x, want)


def test_sets_of_a_captured_batch_come_back_after_the_capture(tc):
    """Each call that the caller captures holds a set until the capture ends; then two of them stay at most."""
    n, steps = 5, 2
    p = tc.Params(n, list(map(float, W.draw_couplings(n, 1))), 1.002, 1.0)
    U = tc.expm_model(p, 0.1)
    rho = torch.from_numpy(W.random_mixed_state(n, 2, 1)[0]).cuda()
    work = torch.empty(1 << 22, dtype=torch.uint8, device="cuda")
    state = rho.clone()
    tc.batch_evolve([U], [state], steps, "fp64", params=[p], inplace=True, observe=False, work=work)
    state.copy_(rho)
    tc.release_idle()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        for _ in range(4):
            tc.batch_evolve([U], [state], steps, "fp64", params=[p], inplace=True, observe=False, work=work)
    tc.batch_evolve([U], [rho], steps, "fp64", params=[p])   # gives its set back: the surplus goes
    assert tc.release_idle() <= 2 and tc.release_idle() == 0
    g.replay()
    want, _ = tc.evolve(U, rho, n, 4 * steps, "fp64", params=p)
    torch.cuda.synchronize()
    assert torch.equal(state, want)

"""Ranked plans of one dimension and different family sizes, side by side: what
one call sets up must not change what another is allowed to launch."""
import threading

import numpy as np
import pytest

import workloads

from gpu_util import run

pytestmark = pytest.mark.gpu

# designs, draws: 512 and 4096 thresholds per coordinate, which take 12 and 98 KB
# of shared memory in one kernel and as many more words in the other
D, SMALL, LARGE = 6, (300, 400_000), (4096, 70_000)


def grid(designs, draws, seed):
    rng = np.random.default_rng(seed)
    return workloads.Problem("ranked", [workloads.lkj_cvine(D, 2.0, rng)], np.zeros(designs, np.int32),
                             list(np.zeros((designs, D))), list(rng.normal(1.2, 0.7, (designs, D))),
                             [draws] * designs, [1] * designs, structures=[{"kind": "dense"}])


@pytest.fixture(scope="module")
def problems():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_10494_gb300 as pkg
    ctx = pkg.Context(0)
    probs = [grid(*SMALL, seed=1), grid(*LARGE, seed=2)]
    return pkg, probs, [run(ctx, p, seed=5)["hits"] for p in probs]


def test_graph_replay_after_a_smaller_plan(problems):
    import torch
    pkg, (small, large), (hits_small, hits_large) = problems
    ctx, s = pkg.Context(0), torch.cuda.Stream()
    big = pkg.Plan(ctx, pkg.DeviceProblem.from_workload(large), shared=True, graph=True)
    little = pkg.Plan(ctx, pkg.DeviceProblem.from_workload(small), shared=True)
    torch.cuda.synchronize()
    first = big.eval(5, stream=s)["hits"]
    other = little.eval(5, stream=s)["hits"]
    s.synchronize()
    np.testing.assert_array_equal(first.cpu().numpy(), hits_large)
    first.zero_()
    torch.cuda.synchronize()
    again = big.eval(5, stream=s)["hits"]
    s.synchronize()
    ctx.sync_status()
    np.testing.assert_array_equal(again.cpu().numpy(), hits_large)
    np.testing.assert_array_equal(other.cpu().numpy(), hits_small)
    big.close()
    little.close()


def test_two_threads_of_different_family_sizes(problems):
    """Calibrations queue many launches in one call, so those of the two threads
    fall between each other's steps; each result equals the one alone."""
    import torch
    pkg, probs, _ = problems
    rng = np.random.default_rng(3)
    jobs = [(pkg.DeviceProblem.from_workload(p),
             torch.as_tensor(rng.dirichlet(np.ones(D), len(p.n_draws)).ravel(), device="cuda")) for p in probs]

    def calibrate(i, stream, ctx):
        dp, w = jobs[i]
        out = pkg.mc_fwer_calibrate(ctx, dp, w, rounds=100, seed=5, stream=stream)
        stream.synchronize()
        ctx.sync_status(stream)
        return {k: v.cpu().numpy() for k, v in out.items()}

    alone = [calibrate(i, torch.cuda.Stream(), pkg.Context(0)) for i in (0, 1)]
    torch.cuda.synchronize()
    failed, got = [], [None, None]
    start = threading.Barrier(2)

    def work(i):
        try:
            torch.cuda.set_device(0)
            ctx, stream = pkg.Context(0), torch.cuda.Stream()
            start.wait(timeout=60)
            for _ in range(20):
                got[i] = calibrate(i, stream, ctx)
        except Exception as e:                          # reported by the test's own thread
            failed.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=120)
    assert not failed, failed
    for i in (0, 1):
        for name, x in alone[i].items():
            np.testing.assert_array_equal(got[i][name], x)

"""The ranked shared-draw path: hit counts bit-identical to the per-design
kernel at the edges of its chunks, families, batches and thresholds."""
import numpy as np
import pytest

import workloads

from gpu_util import run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_10494_gb300 as pkg
    return pkg.Context(0)


def ranked_problem(d, groups, begin, seed):
    """One scenario; groups of (designs, draws) with one stream each.  Thresholds
    with ties, dropped tests, both zeros and a coordinate that no draw exceeds."""
    rng = np.random.default_rng(seed)
    sig = workloads.lkj_cvine(d, 2.0, rng) if d > 1 else np.eye(1)
    mus, bs, n, keys = [], [], [], []
    for g, (m, draws) in enumerate(groups):
        b = rng.normal(1.2, 0.7, (m, d))
        b[:, 0] = np.round(4.0 * b[:, 0]) / 4.0
        b[rng.random((m, d)) < 0.05] = np.inf
        b[rng.random(m) < 0.02, d - 1] = -0.0
        b[rng.random(m) < 0.02, 0] = 0.0
        if d > 2:
            b[:, 1] = np.inf
        mus += list(np.zeros((m, d)))
        bs += list(b)
        n += [draws] * m
        keys += [g] * m
    J = len(n)
    return workloads.Problem("ranked", [sig], np.zeros(J, np.int32), mus, bs, n, keys, draw_begin=np.full(J, begin),
                             structures=[{"kind": "dense"}])


# (dimension, [(designs, draws)], first draw): single and several words per
# row, one more design than a chunk (128, 256, 512) or a family (4096, 2048,
# 1024), one more draw than a batch, offsets inside a group of draws and
# across 2^32 generator calls
CASES = [
    (1, [(32, 1_250_001)], 0),
    (1, [(4097, 80_000), (129, 16_384)], 3),
    (2, [(257, 320_001)], 1),
    (3, [(513, 140_001), (32, 16_385)], 7),
    (3, [(4097, 30_011)], 0),
    (4, [(256, 320_000), (128, 65_537)], (1 << 32) - 70_000),
    (5, [(129, 260_003)], 2),
    (8, [(300, 80_001)], 5),
    (10, [(2049, 20_000), (40, 30_001)], 1),
    (13, [(200, 100_001)], 3),
    (17, [(257, 40_001)], 1),
    (20, [(1025, 16_385), (33, 20_000)], 9),
]


@pytest.mark.parametrize("d,groups,begin", CASES)
def test_ranked_hits_identical_to_per_design(ctx, d, groups, begin):
    work = sum(d * n * -(-m // 256) for m, n in groups)
    assert work >= 1.25e6                                 # the rule that selects the ranked path
    prob = ranked_problem(d, groups, begin, seed=d)
    per = run(ctx, prob, seed=5)
    sh = run(ctx, prob, seed=5, shared=True)
    for name in ("hits", "p", "se"):
        np.testing.assert_array_equal(sh[name], per[name])


def test_ranked_all_below_and_graph_replay(ctx):
    prob = ranked_problem(3, [(700, 150_001)], 4, seed=1)
    per = run(ctx, prob, seed=2, region=1)
    sh = run(ctx, prob, seed=2, region=1, shared=True, graph=True)
    np.testing.assert_array_equal(sh["hits"], per["hits"])


def test_ranked_bad_scenario_and_nan(ctx):
    """A Sigma that is not positive definite gives no hits and MCD_ENOTSPD; a
    NaN threshold is reported and leaves the other designs' counts alone."""
    import paper_2005_10494_gb300 as pkg
    prob = ranked_problem(3, [(64, 500_000)], 0, seed=3)
    good = run(ctx, prob, seed=1)["hits"]
    prob.bs[5] = prob.bs[5].copy()
    prob.bs[5][2] = np.nan
    dp = pkg.DeviceProblem.from_workload(prob)
    plan = pkg.Plan(ctx, dp, shared=True)
    hits = plan.eval(1)["hits"]
    with pytest.raises(pkg.MCDError) as err:
        ctx.sync_status()
    assert err.value.code == 7 and err.value.index == 5
    keep = np.arange(64) != 5
    np.testing.assert_array_equal(hits.cpu().numpy()[keep], good[keep])
    plan.close()
    prob.sigmas[0] = np.array([[1.0, 2.0, 0.0], [2.0, 1.0, 0.0], [0.0, 0.0, 1.0]])
    dp = pkg.DeviceProblem.from_workload(prob)
    plan = pkg.Plan(ctx, dp, shared=True)
    assert int(plan.eval(1)["hits"].sum()) == 0
    with pytest.raises(pkg.MCDError) as err:
        ctx.sync_status()
    assert err.value.code == 2
    plan.close()

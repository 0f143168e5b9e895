"""The ranked shared-draw path where the plan selects it (its kernels run blocks of
512 threads, the direct shared-draw kernel 256): hits bit-identical to the
per-design kernel at the edges of chunks, families, rounds and plans."""
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


def groups_problem(d, groups, begin=0, seed=0, sig=None):
    """One scenario; groups of (designs, draws) with one stream each.  Thresholds
    with ties, dropped tests, both zeros and infinities."""
    rng = np.random.default_rng([d, seed])
    sig = (workloads.lkj_cvine(d, 2.0, rng) if d > 1 else np.eye(1)) if sig is None else sig
    bs, n, keys = [], [], []
    for g, (m, draws) in enumerate(groups):
        b = rng.normal(1.2, 0.7, (m, d))
        b[:, 0] = np.round(4.0 * b[:, 0]) / 4.0
        b[rng.random((m, d)) < 0.03] = np.inf
        b[rng.random(m) < 0.01, d - 1] = -0.0
        b[rng.random(m) < 0.01, 0] = 0.0
        b[rng.random(m) < 0.003, 0] = -np.inf
        bs += list(b)
        n += [draws] * m
        keys += [g] * m
    J = len(n)
    return workloads.Problem("ranked", [sig], np.zeros(J, np.int32), list(np.zeros((J, d))), bs, n, keys,
                             draw_begin=np.full(J, begin), structures=[{"kind": "dense"}])


def threads(ctx, prob, d):
    import paper_2005_10494_gb300 as pkg
    plan = pkg.Plan(ctx, pkg.DeviceProblem.from_workload(prob), shared=True)
    out = plan.config(d)["threads"]
    plan.close()
    return out


# one more design than a chunk (128, 256, 512) or a family (4096, 2048, 1024), one
# more draw than a batch, offsets inside a group of draws and across 2^32
# generator calls; more draws than a round holds (64 MB of ranks), a second group
# behind them; more groups than the 256 families of a round
RANKED = [
    (1, [(32, 4_000_001)], 0),
    (1, [(4097, 600_000), (129, 600_001)], 3),
    (2, [(257, 1_200_001)], 1),
    (3, [(513, 1_000_001), (32, 1_000_000)], 7),
    (3, [(4097, 150_011)], 0),
    (4, [(256, 1_000_000), (128, 600_001)], (1 << 32) - 350_000),
    (5, [(129, 700_003)], 2),
    (8, [(300, 250_001)], 5),
    (10, [(2049, 60_000), (40, 90_001)], 1),
    (13, [(200, 300_001)], 3),
    (17, [(257, 150_001)], 1),
    (20, [(1025, 50_001), (33, 50_000)], 9),
    (20, [(32, 1_900_003), (40, 700_001)], 6),
    (4, [(33, 9_000_001), (64, 100_001)], 3),
    (3, [(33, 40_003)] * 300, 1),
]


@pytest.mark.parametrize("d,groups,begin", RANKED)
def test_ranked_where_selected(ctx, d, groups, begin):
    prob = groups_problem(d, groups, begin)
    assert threads(ctx, prob, d) == 512
    per, sh = run(ctx, prob, seed=5), run(ctx, prob, seed=5, shared=True)
    for name in ("hits", "p", "se"):
        np.testing.assert_array_equal(sh[name], per[name])


@pytest.mark.parametrize("d,designs,draws", [(3, 2600, 16_383), (3, 1100, 50_001), (20, 600, 12_001)])
def test_direct_kernel_below_the_rule(ctx, d, designs, draws):
    """Several chunks, ragged draws: too little work for ranks."""
    prob = groups_problem(d, [(designs, draws)], begin=2, seed=1)
    assert threads(ctx, prob, d) == 256
    np.testing.assert_array_equal(run(ctx, prob, seed=5, shared=True)["hits"], run(ctx, prob, seed=5)["hits"])


def test_all_kinds_of_groups_in_one_plan(ctx):
    """Ranked and direct groups of two dimensions and designs with a stream of
    their own, in one launch sequence, directly and replayed from a graph."""
    parts = [groups_problem(3, [(600, 1_000_000), (40, 5_001), (5, 70_001)], seed=2),
             groups_problem(10, [(300, 300_001), (100, 9_999), (31, 20_000)], seed=3)]
    assert threads(ctx, parts[0].subset(range(600)), 3) == 512
    assert threads(ctx, parts[1].subset(range(300)), 10) == 512
    prob = workloads.Problem("kinds", [p.sigmas[0] for p in parts],
                             np.concatenate([np.full(len(p.n_draws), s) for s, p in enumerate(parts)]).astype(np.int32),
                             sum((list(p.mus) for p in parts), []), sum((list(p.bs) for p in parts), []),
                             np.concatenate([p.n_draws for p in parts]), np.concatenate([p.keys for p in parts]),
                             structures=[{"kind": "dense"}] * 2)
    per = run(ctx, prob, seed=5)["hits"]
    np.testing.assert_array_equal(run(ctx, prob, seed=5, shared=True)["hits"], per)
    np.testing.assert_array_equal(run(ctx, prob, seed=5, shared=True, graph=True)["hits"], per)


def test_ranked_failures_where_selected(ctx):
    """NaN thresholds and a Sigma that is not positive definite."""
    import paper_2005_10494_gb300 as pkg
    prob = groups_problem(3, [(64, 2_000_000)], seed=4)
    assert threads(ctx, prob, 3) == 512
    good = run(ctx, prob, seed=1)["hits"]
    prob.bs[5] = np.array([1.0, 1.0, np.nan])
    plan = pkg.Plan(ctx, pkg.DeviceProblem.from_workload(prob), shared=True)
    hits = plan.eval(1)["hits"]
    with pytest.raises(pkg.MCDError) as err:
        ctx.sync_status()
    assert err.value.code == 7 and err.value.index == 5
    keep = np.arange(64) != 5
    np.testing.assert_array_equal(hits.cpu().numpy()[keep], good[keep])
    plan.close()
    bad = groups_problem(3, [(64, 2_000_000)], seed=4, sig=np.array([[1.0, 2.0, 0.0], [2.0, 1.0, 0.0], [0.0, 0.0, 1.0]]))
    plan = pkg.Plan(ctx, pkg.DeviceProblem.from_workload(bad), shared=True)
    assert int(plan.eval(1)["hits"].sum()) == 0
    with pytest.raises(pkg.MCDError) as err:
        ctx.sync_status()
    assert err.value.code == 2
    plan.close()

"""The boxed adjoint against the direct test of every design, in the same order:
the same bits in hits, likelihood-ratio and sigmoid gradients."""
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


def problem(d, groups, seed, lo=1.0, hi=2.5):
    """Groups of (designs, draws), neighbours on a line of thresholds."""
    rng = np.random.default_rng([d, seed])
    sig = workloads.lkj_cvine(d, 2.0, rng)
    bs, n, keys = [], [], []
    for g, (m, draws) in enumerate(groups):
        u = rng.uniform(-0.5, 0.5, d)
        bs.append(rng.uniform(lo, hi, d) + np.linspace(0.0, 1.0, m)[:, None] * u)
        n += [draws] * m
        keys += [g + 1] * m
    b = np.concatenate(bs)
    J = len(n)
    return workloads.Problem("boxed", [sig], np.zeros(J, np.int32), list(np.zeros((J, d))), list(b), n, keys,
                             structures=[{"kind": "dense"}])


@pytest.mark.parametrize("d", [11, 12])
@pytest.mark.parametrize("designs", [33, 250, 600])
@pytest.mark.parametrize("h", [0.0, 0.02])
def test_kernels_agree_bit_for_bit(ctx, d, designs, h):
    """A plan with fewer tiles than resident blocks takes the direct kernel, and
    with a second group the boxed one: same tiles, same slots of the first group."""
    draws = 60_001 if d == 11 else 15_001
    one = run(ctx, problem(d, [(designs, draws)], 0), seed=4, grad=True, k=0, h=h, shared=True)
    two = run(ctx, problem(d, [(designs, draws), (40, 400_000)], 0), seed=4, grad=True, k=0, h=h, shared=True)
    for name in ("hits", "grad_lr", "grad_sig", "grad_se"):
        if name in one:
            a = one[name].ravel()
            np.testing.assert_array_equal(a, two[name].ravel()[:a.size])


@pytest.mark.parametrize("d,draws", [(10, 4_000_000), (11, 400_003), (12, 90_001), (17, 30_001), (18, 40_000), (19, 10_001),
                                     (20, 30_001)])
@pytest.mark.parametrize("h", [0.0, 0.02])
def test_fallback_agrees_bit_for_bit(ctx, d, draws, h):
    """The last design of each word of 32 decides the path of the other 31: dropped
    tests (+inf, as good as absent) or its neighbour's thresholds leave the box
    narrow, thresholds that every draw exceeds make every draw a tested one, so
    that the warp takes the direct loop."""
    prob = problem(d, [(224, draws)], 1, 2.0, 3.2)
    last = np.arange(31, 224, 32)
    keep = np.setdiff1d(np.arange(224), last)
    out = []
    for how in ("absent", "neighbour", "wide"):
        bs = [b.copy() for b in prob.bs]
        for j in last:
            bs[j] = np.full(d, np.inf) if how == "absent" else bs[j - 1].copy() if how == "neighbour" else np.full(d, -np.inf)
        prob.bs, keep_bs = bs, prob.bs
        out.append(run(ctx, prob, seed=4, grad=True, k=0, h=h, shared=True))
        prob.bs = keep_bs
    assert (out[2]["hits"][last] == draws).all() and (out[0]["hits"][last] == 0).all()
    assert (out[0]["hits"][keep] > 0).all()
    for other in out[1:]:
        np.testing.assert_array_equal(out[0]["hits"][keep], other["hits"][keep])
        for name in ("grad_lr", "grad_sig", "grad_se"):
            if name in other:
                np.testing.assert_array_equal(out[0][name].reshape(224, d)[keep], other[name].reshape(224, d)[keep])


@pytest.mark.parametrize("d,designs,draws", [(9, 33, 70_001), (10, 65, 20_000), (13, 40, 9_001), (16, 97, 30_001)])
def test_warps_without_designs(ctx, d, designs, draws):
    """A chunk that leaves warps empty: hits as the per-design kernel's, gradients
    within the rounding of its FP32 sums."""
    prob = problem(d, [(designs, draws)], 2)
    a = run(ctx, prob, seed=4, grad=True, k=0, h=0.02, shared=True)
    b = run(ctx, prob, seed=4, grad=True, k=0, h=0.02)
    np.testing.assert_array_equal(a["hits"], b["hits"])
    np.testing.assert_allclose(a["grad_lr"], b["grad_lr"], rtol=0, atol=2e-5 * np.abs(b["grad_lr"]).max() + 1e-5)

"""Gradient finalisation of designs of several dimensions in one launch, and of a
design whose slot sums may pass 63 bits."""
import math

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


@pytest.mark.parametrize("k", [0, 3])
@pytest.mark.parametrize("designs,draws", [(3, 900), (40, 1_500_000), (900, 900), (900, 70_000), (30_000, 900)])
def test_mixed_dimensions_match_each_dimension_alone(ctx, designs, draws, k):
    """Above d = 10 each dimension has its sampling kernel in either plan, so the
    slot sums are the same whole numbers and the results differ by the rounding
    of a triangular solve, below 1e-13 times a condition number of at most 1e3,
    and of at most 32 FP64 additions.  Draws fill one slot, some or all 32."""
    rng = np.random.default_rng(designs + k)
    dims = list(range(11, 21))
    sigs = [0.5 * np.eye(d) + 0.5 * np.ones((d, d)) for d in dims]
    scen = rng.integers(0, len(dims), designs).astype(np.int32)
    scen[0], scen[-1] = 0, len(dims) - 1
    mus = [np.zeros(dims[s]) for s in scen]
    bs = [rng.normal(1.5, 0.4, dims[s]) for s in scen]
    prob = workloads.Problem("mixed", sigs, scen, mus, bs, [draws] * designs, np.arange(designs),
                             structures=[{"kind": "dense"}] * len(dims))
    width = np.array([dims[s] for s in scen])
    at = np.concatenate([[0], np.cumsum(width)])
    jac = rng.normal(size=(int(at[-1]), k)) if k else None
    both = run(ctx, prob, seed=3, grad=True, k=k, jac=jac, h=0.05)
    for s in sorted(set(scen.tolist())):
        idx = np.flatnonzero(scen == s)
        rows = np.concatenate([np.arange(at[j], at[j + 1]) for j in idx])
        one = run(ctx, prob.subset(idx), seed=3, grad=True, k=k, jac=None if jac is None else jac[rows], h=0.05)
        np.testing.assert_array_equal(one["hits"], both["hits"][idx])
        for name in ("grad_lr", "grad_sig"):
            a = one[name].ravel()
            b = both[name].reshape(designs, k)[idx].ravel() if k else both[name].ravel()[rows]
            scale = np.sqrt(np.mean(a * a))
            assert scale > 0 and np.abs(a - b).max() <= 1e-10 * max(scale, np.abs(a).max())
        se = both["grad_se"].reshape(designs, k)[idx] if k else both["grad_se"].ravel()[rows]
        assert np.isnan(se).all() if draws == 900 else (se > 0).all()


def test_gradient_beyond_32_bits_of_draws(ctx):
    """d = 1, more than 2^32 draws beside a design of few: dp/dmu is the normal
    density at the threshold; the FP32 normals move it by less than 1e-5."""
    b, n = 0.7, (1 << 32) + 12_345
    prob = workloads.Problem("many draws", [np.eye(1)], np.zeros(2, np.int32), [np.zeros(1)] * 2, [np.full(1, b)] * 2,
                             [n, 50_000], [1, 2], structures=[{"kind": "dense"}])
    out = run(ctx, prob, seed=7, grad=True, k=0)
    g, se = out["grad_lr"].ravel(), out["grad_se"].ravel()
    exact = math.exp(-0.5 * b * b) / math.sqrt(2.0 * math.pi)
    spread = math.sqrt(out["p"][0] / n)                  # of the mean of 1_R z, up to a factor of order one
    assert 0.2 * spread < se[0] < 5.0 * spread
    assert abs(g[0] - exact) < 6.0 * se[0] + 1e-5
    assert abs(g[1] - exact) < 10.0 / math.sqrt(50_000)

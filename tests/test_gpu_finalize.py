"""Gradient finalisation on either side of the sizes at which the number of
lanes per design changes."""
import numpy as np
import pytest

import workloads

from gpu_util import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [0, 2])
@pytest.mark.parametrize("many,most", [(2048, 20_000), (2048, 400_000), (16384, 20_000), (16384, 400_000)])
def test_gradients_either_side_of_a_lane_change(many, most, k):
    """The same designs in a plan of many - 1 and in one of many (with one more
    design of a few draws): the slot sums are the same whole numbers, so the
    results differ by the order of at most 32 FP64 additions and by the
    rounding of two triangular solves, below 1e-13 times a condition number of
    at most 1e3.  Designs of up to 20,000 draws fill one slot (no standard
    error), those of up to 400,000 several."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_10494_gb300 as pkg
    ctx = pkg.Context(0)
    rng = np.random.default_rng(many)
    dims = [1, 3, 10]
    sigs = [0.5 * np.eye(d) + 0.5 * np.ones((d, d)) for d in dims]
    scen = np.append(rng.integers(0, 3, many - 1), 1).astype(np.int32)
    mus = [np.zeros(dims[s]) for s in scen]
    bs = [rng.normal(1.3, 0.4, dims[s]) for s in scen]
    n = np.append(rng.integers(1, most + 1, many - 1), 100)
    prob = workloads.Problem("finalize", sigs, scen, mus, bs, n, np.arange(many),
                             structures=[{"kind": "dense"}] * 3)
    width = sum(len(m) for m in mus)
    jac = rng.normal(size=(width, k)) if k else None
    big = run(ctx, prob, seed=3, grad=True, k=k, jac=jac, h=0.05)
    cut = width - dims[scen[-1]]
    small = run(ctx, prob.subset(range(many - 1)), seed=3, grad=True, k=k, jac=None if jac is None else jac[:cut], h=0.05)
    np.testing.assert_array_equal(small["hits"], big["hits"][:many - 1])
    for name in ("grad_lr", "grad_sig", "grad_se"):
        a = small[name].ravel()
        b = big[name].ravel()[:a.size]
        np.testing.assert_array_equal(np.isnan(a), np.isnan(b))
        fine = ~np.isnan(a)
        assert fine.sum() > a.size // 2 or (name == "grad_se" and most == 20_000)
        if not fine.any():
            continue
        rms = np.sqrt(np.mean(a[fine] ** 2))
        assert np.abs(a - b)[fine].max() <= 1e-10 * max(rms, np.abs(a[fine]).max())

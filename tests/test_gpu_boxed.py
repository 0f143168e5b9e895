"""The boxed shared-draw adjoint: neighbouring designs (whole words of a box
agree) against the same designs in a random order (draw by draw)."""
import numpy as np
import pytest

import workloads

from gpu_util import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,designs,draws,begin", [(9, 257, 70_001, 3), (10, 1024, 90_000, 0), (11, 33, 50_003, 1),
                                                   (12, 300, 40_001, (1 << 32) - 20_000), (14, 600, 33_333, 5),
                                                   (17, 129, 30_001, 2), (20, 512, 25_600, 0), (20, 90, 1_000, 7)])
@pytest.mark.parametrize("h", [0.0, 0.02])
def test_boxed_adjoint_of_neighbours_and_of_a_shuffle(d, designs, draws, begin, h):
    """Hits and the sums A and B do not depend on the neighbours: the counts and
    grad_lr are the same bits.  The sigmoid sums take terms below 3e-8 or not
    with the neighbours, and round with them."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_10494_gb300 as pkg
    ctx = pkg.Context(0)
    rng = np.random.default_rng(d + designs)
    sig = workloads.lkj_cvine(d, 2.0, rng)
    u = rng.uniform(-0.5, 0.5, d)
    b = rng.uniform(1.0, 2.5, d) + np.linspace(0.0, 1.0, designs)[:, None] * u
    b[rng.random((designs, d)) < 0.01] = np.inf
    b[0, 0] = -np.inf
    out = []
    order = rng.permutation(designs)
    for idx in (np.arange(designs), order):
        prob = workloads.Problem("boxed", [sig], np.zeros(designs, np.int32), list(np.zeros((designs, d))), list(b[idx]),
                                 [draws] * designs, [1] * designs, draw_begin=np.full(designs, begin),
                                 structures=[{"kind": "dense"}])
        out.append(run(ctx, prob, seed=4, grad=True, k=0, h=h, shared=True))
    a, s = out
    np.testing.assert_array_equal(a["hits"][order], s["hits"])
    g = {name: x.reshape(designs, d) for name, x in a.items() if name.startswith("grad")}
    np.testing.assert_array_equal(g["grad_lr"][order].ravel(), s["grad_lr"].ravel())
    if h:
        np.testing.assert_allclose(g["grad_sig"][order].ravel(), s["grad_sig"].ravel(), rtol=2e-3, atol=2e-4)

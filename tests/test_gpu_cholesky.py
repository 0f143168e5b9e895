"""The factorisation by warps and by threads: the same scenarios in a plan of few
and in one of many give the same counts, and the same failures."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,many", [(1, 1500), (5, 2500), (6, 461), (10, 1381), (20, 3681)])
def test_few_and_many_scenarios_agree(d, many):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_10494_gb300 as pkg
    ctx = pkg.Context(0)
    rng = np.random.default_rng(d)
    few = 40
    sigs = [workloads.lkj_cvine(d, 2.0, rng) if d > 1 else np.array([[rng.uniform(0.5, 2.0)]]) for _ in range(few)]
    sigs[7] = sigs[7].copy()
    sigs[7][d - 1, d - 1] = 0.0                          # not positive definite
    t = list(rng.normal(1.0, 0.5, (few, d)))

    def hits(n):
        prob = workloads.Problem("scenarios", [sigs[s % few] for s in range(n)], np.arange(n, dtype=np.int32),
                                 [np.zeros(d)] * n, [t[s % few] for s in range(n)], [4001] * n,
                                 [s % few for s in range(n)], structures=[{"kind": "dense"}] * n)
        plan = pkg.Plan(ctx, pkg.DeviceProblem.from_workload(prob))
        out = plan.eval(3)["hits"].cpu().numpy()
        with pytest.raises(pkg.MCDError) as err:
            ctx.sync_status()
        assert err.value.code == 2 and err.value.index % few == 7
        plan.close()
        return out

    a = hits(few)
    assert a[7] == 0 and (np.delete(a, 7) > 0).all()
    np.testing.assert_array_equal(hits(many), a[np.arange(many) % few])

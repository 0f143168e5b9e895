"""Draw counts that no plan can schedule are refused with an argument error before
any table is built."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,designs,draws", [(3, 32, 1 << 50), (1, 4096, 1 << 55), (20, 40, 1 << 52)])
@pytest.mark.parametrize("shared", [True, False])
def test_too_many_draws_are_refused(d, designs, draws, shared):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_10494_gb300 as pkg
    ctx = pkg.Context(0)
    prob = workloads.Problem("limits", [np.eye(d)], np.zeros(designs, np.int32), list(np.zeros((designs, d))),
                             list(np.ones((designs, d))), [draws] * designs, [1] * designs,
                             structures=[{"kind": "dense"}])
    dp = pkg.DeviceProblem.from_workload(prob)
    free = torch.cuda.mem_get_info()[0]
    with pytest.raises(pkg.MCDError) as err:
        pkg.Plan(ctx, dp, shared=shared)
    assert err.value.code == 1 and "too many tiles" in str(err.value)
    assert torch.cuda.mem_get_info()[0] >= free - (64 << 20)

"""The event profiler has one record per kernel launch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2207_00426_gb300 import workloads as W


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("n,sums", [(3 * 2048, 1), (3 * 2048 + 1, 2)])
def test_one_record_per_launch(graph, n, sums):
    """Three steps per leaf: up to 2048 leaf chunks the log-likelihood is one
    launch, beyond two; a solve's own launches are the prior's broadcast, its
    deviation and the conversion of the result."""
    from paper_2207_00426_gb300 import binding as B
    d = W.ct_batch(lengths=[n], seed=8)
    y, m0, N0 = (torch.tensor(np.ascontiguousarray(d[k]), dtype=torch.float32, device="cuda:0")
                 for k in ("y", "m0", "N0"))
    ctx = B.Context(0, use_graph=graph)
    ctx.profile(True)
    B.sqsm_ipls_smooth(ctx, d["theta"], y, d["offsets"], m0, N0, 2, B.EXTENDED, dt=d["dt"])
    torch.cuda.synchronize()
    count = {k: c for k, (_, c) in ctx.profile_read().items()}
    ctx.close()
    assert count["loglik_reduce"] == sums and count["broadcast_prior"] == 3
    assert count["ct_slr"] == 2 and count["smoother_leaf_down"] == 2

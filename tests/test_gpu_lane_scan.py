"""FP64 upper scan levels with a combine spread over lanes (chunks of 8 / 16
items, folds of 4, folds per thread above 20000 items): the default context
against one whose explicit radix takes the one-thread and one-warp folds, at
sizes around the chunks, the folds and the changes of form.  Both sides are
backward-stable FP64 evaluations of the same recursion, so they agree to the
parity tolerance of the FP64 build (1e-9)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2207_00426_gb300 import workloads as W
from gpu_util import rel_mean_err, rel_cov_err, TOL


@pytest.fixture(scope="module")
def B():
    from paper_2207_00426_gb300 import binding
    return binding


def _compare(a, b):
    a, b = [[v.cpu().numpy() for v in r] for r in (a, b)]
    t = TOL["f64"]
    assert rel_mean_err(a[0], b[0]) < t["mean"] and rel_cov_err(a[1], b[1]) < t["cov"]
    assert np.all(np.isfinite(a[1])) and np.all(np.diagonal(a[1], axis1=1, axis2=2) >= 0)


@pytest.mark.parametrize("nx,ny", [(3, 2), (4, 2), (5, 2), (6, 3)])
@pytest.mark.parametrize("n", [1, 2, 8, 9, 16, 17, 65, 513, 4864, 4866])
def test_linear(B, nx, ny, n):
    m = W.random_lgssm(n, nx, ny, seed=n + 10 * nx)
    q = {k: torch.tensor(np.ascontiguousarray(v), device="cuda:0") for k, v in m.items() if k != "x"}
    r = [B.sqsm_lgssm_smooth(c, q["F"], q["c"], q["SQ"], q["H"], q["d"], q["SR"], q["m0"], q["N0"],
                             q["y"]) for c in (B.Context(0), B.Context(0, leaf_chunk=3, radix=4))]
    torch.cuda.synchronize()
    _compare(r[0][:2], r[1][:2])
    _compare(r[0][2:4], r[1][2:4])
    assert abs(r[0][4].item() - r[1][4].item()) <= 1e-10 * abs(r[1][4].item())


@pytest.mark.parametrize("lengths", [[1, 2, 9, 300, 8, 17], [45_000]])
def test_tracks(B, lengths):
    """Ragged batch, and a track whose first upper level is folded per thread
    (22500 items)."""
    d = W.ct_batch(batch=len(lengths), lengths=lengths, seed=11)
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda:0")
    r = [B.sqsm_ipls_smooth(c, d["theta"], t(d["y"]), d["offsets"], t(d["m0"]), t(d["N0"]), 1)
         for c in (B.Context(0), B.Context(0, leaf_chunk=3, radix=4))]
    torch.cuda.synchronize()
    _compare(r[0][:2], r[1][:2])

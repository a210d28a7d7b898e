"""A NaN in an input reaches the results of the steps that depend on it: the
factorisation's structural zeros leave out products with exact zeros, never a
row's own entry."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2207_00426_gb300 import workloads as W


@pytest.fixture(scope="module")
def B():
    from paper_2207_00426_gb300 import binding
    return binding


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("nx,ny", [(3, 2), (5, 2), (2, 3)])
@pytest.mark.parametrize("n,leaf", [(1, 0), (6, 0), (200, 0), (200, 200)])
@pytest.mark.parametrize("key", ["SQ", "SR"])
def test_nan_in_last_noise_entry(B, dt, nx, ny, n, leaf, key):
    """The last diagonal entry of step k's S_Q (S_R), which no other row of
    the factor shares: P^- (S) of that step is NaN in plain arithmetic, so
    its gain, its log-likelihood and every filtering mean from k on are."""
    m = W.random_lgssm(n, nx, ny, seed=3)
    k = n // 2
    m[key][k, -1, -1] = np.nan
    q = {a: torch.tensor(v, dtype=dt, device="cuda:0") for a, v in m.items() if a != "x"}
    ctx = B.Context(0, leaf_chunk=leaf)
    mf, Nf, ms, Ns, ll = B.sqsm_lgssm_smooth(ctx, q["F"], q["c"], q["SQ"], q["H"], q["d"], q["SR"],
                                             q["m0"], q["N0"], q["y"])
    torch.cuda.synchronize()
    assert bool(torch.isfinite(mf[: k + 1]).all()) and bool(torch.isfinite(Nf[: k + 1]).all())
    assert bool(torch.isnan(mf[k + 1:]).all())
    assert bool(torch.isnan(Nf[k + 1:]).flatten(1).any(1).all())
    assert bool(torch.isnan(ll).all())
    assert ctx.status() & B.ERR_NONFINITE
    ctx.close()

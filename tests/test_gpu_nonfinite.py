"""A NaN in an input reaches the results of the steps that depend on it: the
factorisation's structural zeros leave out products with exact zeros, never a
row's own entry.  A difference of sigma points that overflows divides to
infinity."""
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


@pytest.mark.parametrize("rule", ["CUBATURE", "UNSCENTED"])
def test_overflowing_difference_stays_infinite(B, rule):
    """FP64, a turn of 1 rad per step and a spread of 7e307 of v_x: the points'
    v_y are +- s sin(1) 7e307 (s^2 = 5 or 6), both finite; their difference
    overflows, and the regression's F[v_y][v_x] = inf / (2 s) / 7e307 is
    infinite."""
    f64, big = torch.float64, 7e307
    ms = torch.zeros((2, 5), dtype=f64, device="cuda:0")
    ms[:, 4] = 100.0                    # dt = 0.01
    Ns = 1e-3 * torch.eye(5, dtype=f64, device="cuda:0").repeat(2, 1, 1)
    Ns[0, 2, 2] = big
    F = B.sqsm_ct_linearize(B.Context(0), W.CT_THETA_TRUE,
                            torch.zeros((1, 2), dtype=f64, device="cuda:0"), [0, 1], ms, Ns,
                            getattr(B, rule))[0]
    torch.cuda.synchronize()
    assert F[0, 3, 2].item() == float("inf")

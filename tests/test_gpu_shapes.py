"""Small launches of the smoothers' bookkeeping at the sizes where they change:
conversion of state rows (blocks of 128), the log-likelihood's sum in slices
of 2048 chunks, the default leaf at the lengths where it changes, the
Gauss-Hermite regression with 16 lanes per step."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2207_00426_gb300 import workloads as W


@pytest.fixture(scope="module")
def B():
    from paper_2207_00426_gb300 import binding
    return binding


def _t(a, dt):
    return torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda:0")


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("lengths", [[1], [126], [127], [128], [255, 1, 3]])
def test_rows_conversion_is_exact(B, dt, lengths):
    """Two iterations equal one iteration and another from its result, bit for
    bit: the caller's rows and the packed ones hold the same numbers."""
    d = W.ct_batch(batch=len(lengths), lengths=lengths, seed=5)
    ctx = B.Context(0)
    a = (ctx, d["theta"], _t(d["y"], dt), d["offsets"], _t(d["m0"], dt), _t(d["N0"], dt))
    two = B.sqsm_ipls_smooth(*a, 2)
    one = B.sqsm_ipls_smooth(*a, 1)
    junk = one[1] + torch.triu(torch.ones(5, 5, dtype=dt, device="cuda:0"), 1)   # ignored part
    again = B.sqsm_ipls_smooth(*a, 1, init_ms=one[0], init_Ns=junk)
    torch.cuda.synchronize()
    for u, v in zip(two, again):
        assert torch.equal(u, v)
    assert torch.equal(two[1], torch.tril(two[1]))


@pytest.mark.parametrize("n", [2048, 2049, 6145, 16384])
def test_loglik_in_slices(B, n):
    """One step per leaf: the sum of n partial values in slices of 2048 against
    one chunk per sequence (a single running FP64 sum): both round each of
    their n additions, so they differ by at most 2 n u of the absolute sum."""
    m = W.linear_cv(n=n, seed=3)
    q = {k: _t(v, torch.float64) for k, v in m.items() if k != "x"}
    ll = [B.sqsm_lgssm_smooth(c, q["F"], q["c"], q["SQ"], q["H"], q["d"], q["SR"], q["m0"],
                              q["N0"], q["y"])[4].item()
          for c in (B.Context(0, leaf_chunk=1), B.Context(0, leaf_chunk=n))]
    # every step's term is below 20 in magnitude here; recursion rounding 1e-10
    assert abs(ll[0] - ll[1]) <= 2 * n * 2.0 ** -53 * 20 * n + 1e-10 * abs(ll[1])


@pytest.mark.parametrize("nx,dt,n,leaf", [
    (5, torch.float32, 1, 3), (5, torch.float32, 116_736, 3), (5, torch.float32, 116_737, 4),
    (5, torch.float64, 1, 1), (5, torch.float64, 16_384, 1), (5, torch.float64, 16_385, 2),
    (5, torch.float64, 65_536, 2), (5, torch.float64, 65_537, 3),
    (1, torch.float32, 4096, 1), (1, torch.float32, 4097, 2), (1, torch.float32, 12_289, 3)])
def test_default_leaf(B, nx, dt, n, leaf):
    """The default context gives the bits of one with the leaf spelt out."""
    if nx == 5:
        if torch.cuda.get_device_properties(0).multi_processor_count == 152:
            assert B.Context(0).scan_shape([0, n], dt) == (leaf, 0)
        return
    d = W.ricker_batch([n], seed=3)
    r = [B.sqsm_ipls_smooth_population(c, d["theta"], _t(d["y"], dt), d["offsets"],
                                       _t(d["m0"], dt), _t(d["N0"], dt), 2)
         for c in (B.Context(0), B.Context(0, leaf_chunk=leaf))]
    torch.cuda.synchronize()
    for u, v in zip(*r):
        assert torch.equal(u, v)


@pytest.mark.parametrize("lengths", [[1], [7], [8], [9, 1, 30], [200]])
def test_gauss_hermite_lanes(B, lengths):
    """FP32 (16 lanes per step) against the FP64 build (one thread per step)
    of the same regression: sums of 243 FP32 terms, 243 u = 1.5e-5 of the
    largest term at most."""
    d = W.ct_batch(batch=len(lengths), lengths=lengths, seed=8)
    rng = np.random.default_rng(2)
    rows = int(d["offsets"][-1]) + len(lengths)
    ms = np.concatenate([np.tile(m, (k + 1, 1)) for m, k in zip(d["m0"], lengths)])
    ms = ms + 0.1 * rng.standard_normal(ms.shape)
    Ns = np.tril(0.05 * rng.standard_normal((rows, 5, 5))) + 0.2 * np.eye(5)
    ms, Ns = ms.astype(np.float32), Ns.astype(np.float32)
    out = [[v.double().cpu().numpy() for v in
            B.sqsm_ct_linearize(B.Context(0), d["theta"], _t(d["y"].astype(np.float32), dt),
                                d["offsets"], _t(ms, dt), _t(Ns, dt), B.GAUSS_HERMITE)]
           for dt in (torch.float32, torch.float64)]
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 243 * 2.0 ** -24 * max(1.0, np.abs(b).max()) * 4

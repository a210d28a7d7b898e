"""The Gauss-Hermite regression with 16 lanes per step."""
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

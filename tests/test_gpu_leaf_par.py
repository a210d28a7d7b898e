"""FP32 leaf kernels with the steps of a chunk side by side (chunks of 3, blocks
of 32 chunks, calls of up to 16384 chunks), at the sizes where the last chunk
or block is short."""
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


def _t(a, dt=torch.float32):
    return torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda:0")


@pytest.mark.parametrize("n,options", [(1, {}), (2, {}), (3, dict(absolute=True)), (95, {}),
                                       (97, dict(absolute=True)), (98, dict(refine=1))])
def test_tracks_equal_the_serial_leaf(B, n, options):
    """The same sequence alone and in a batch of more than 16384 chunks, which
    takes one thread per chunk: the same operations in the same order, bit for
    bit."""
    k = 16384 // ((n + 2) // 3) + 1
    d = W.ct_batch(batch=1, lengths=[n], seed=4)
    one = (_t(d["y"]), d["offsets"], _t(d["m0"]), _t(d["N0"]))
    many = (one[0].repeat(k, 1), np.arange(k + 1) * n, one[2].repeat(k, 1), one[3].repeat(k, 1, 1))
    r = [B.sqsm_ipls_smooth(B.Context(0, **options), d["theta"], *a, 3) for a in (one, many)]
    torch.cuda.synchronize()
    for a, b in zip(r[0][:2], r[1][:2]):
        assert torch.equal(a, b[:n + 1]) and torch.equal(a, b[-n - 1:])


@pytest.mark.parametrize("nx,ny", [(3, 2), (4, 2), (5, 2), (6, 3)])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 96, 97, 98, 3073, 49_150])
def test_linear(B, nx, ny, n):
    """Against leaves of four steps, one thread per chunk: either side is within
    the FP32 parity tolerance of the exact result, so they are within twice."""
    m = W.random_lgssm(n, nx, ny, seed=n + 10 * nx)
    q = {k: _t(v) for k, v in m.items() if k != "x"}
    r = [[v.double().cpu().numpy() for v in
          B.sqsm_lgssm_smooth(c, q["F"], q["c"], q["SQ"], q["H"], q["d"], q["SR"], q["m0"],
                              q["N0"], q["y"])] for c in (B.Context(0), B.Context(0, leaf_chunk=4))]
    t = TOL["f32"]
    for i in (0, 2):
        assert rel_mean_err(r[0][i], r[1][i]) < 2 * t["mean"]
        assert rel_cov_err(r[0][i + 1], r[1][i + 1]) < 2 * t["cov"]
    assert abs(r[0][4] - r[1][4]) <= 2 * t["ll"] * abs(r[1][4])

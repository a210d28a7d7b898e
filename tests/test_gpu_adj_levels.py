"""The adjoint's scans in FP64 have levels of their own, apart from the
filter's lane forms: the gradient at the edges of their chunks (32 items, one
or two steps each) against scans folded 4 items at a time."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2207_00426_gb300 import workloads as W


@pytest.mark.parametrize("lengths", [[1], [2, 1, 1], [32], [33], [1024], [1025], [40, 1, 300],
                                     [1024] * 3 + [1], [1] * 40 + [33], [16384], [16385],
                                     [4000] * 10, [4000] * 10 + [2], [999] * 90])
def test_fp64_gradient_against_folded_levels(lengths):
    from paper_2207_00426_gb300 import binding as B
    f64 = torch.float64
    d = W.ct_batch(lengths=lengths, seed=11)
    y, m0, N0 = (torch.tensor(np.ascontiguousarray(d[k]), dtype=f64, device="cuda:0")
                 for k in ("y", "m0", "N0"))
    r = []
    for ctx in (B.Context(0), B.Context(0, leaf_chunk=4, radix=4)):
        nll, g, _, _, _ = B.sqsm_ipls_nll_grad(ctx, d["theta"], y, d["offsets"], m0, N0, 2, 3,
                                               dt=d["dt"], linearization=B.EXTENDED)
        torch.cuda.synchronize()
        assert ctx.status() == 0
        r.append((nll.item(), g.cpu().numpy()))
        ctx.close()
    # another bracketing of the same scans: FP64 rounding, as in the other
    # comparisons of gradients under two scan shapes
    assert abs(r[0][0] - r[1][0]) <= 1e-10 * abs(r[1][0])
    np.testing.assert_allclose(r[0][1], r[1][1], rtol=1e-8, atol=1e-8 * np.abs(r[1][1]).max())

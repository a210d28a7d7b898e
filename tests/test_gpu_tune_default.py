"""The default scan shape is among the shapes the autotuner times."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2207_00426_gb300 import workloads as W


@pytest.mark.parametrize("n", [512, 4000])
def test_autotuned_fp64_keeps_one_step_per_leaf(n):
    """One step per leaf takes four fifths of the time of the next shape at
    these lengths (FP64), far beyond the timing's spread."""
    from paper_2207_00426_gb300 import binding as B
    f64 = torch.float64
    d = W.ct_batch(lengths=[n], seed=7)
    a = [torch.tensor(np.ascontiguousarray(d[k]), dtype=f64, device="cuda:0")
         for k in ("y", "m0", "N0")]
    tuned, plain = B.Context(0, autotune=True), B.Context(0)
    rt, rp = [B.sqsm_ipls_smooth(c, d["theta"], a[0], d["offsets"], a[1], a[2], 3, dt=d["dt"])
              for c in (tuned, plain)]
    torch.cuda.synchronize()
    assert plain.scan_shape(d["offsets"], f64) == (1, 0)
    assert tuned.scan_shape(d["offsets"], f64) == (1, 0)
    for u, v in zip(rt, rp):
        assert torch.equal(u, v)
    tuned.close()
    plain.close()

"""The scan shape that a query reports is the one the calls run with, for every
kind of model."""
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
@pytest.mark.parametrize("n", [100, 4000, 4097, 10_000, 12_289])
def test_population_calls_run_the_reported_shape(B, dt, n):
    """Bit for bit the same with the reported leaf spelt out, and another leaf
    gives other bits somewhere (so the comparison can tell)."""
    d = W.ricker_batch([n], seed=3)
    a = (d["theta"], _t(d["y"], dt), d["offsets"], _t(d["m0"], dt), _t(d["N0"], dt), 3)
    plain = B.Context(0)
    leaf, radix = plain.scan_shape(d["offsets"], dt, model=B.MODEL_POPULATION)
    assert radix == 0
    r = [B.sqsm_ipls_smooth_population(c, *a)
         for c in (plain, B.Context(0, leaf_chunk=leaf), B.Context(0, leaf_chunk=leaf + 1))]
    torch.cuda.synchronize()
    assert all(torch.equal(u, v) for u, v in zip(r[0], r[1]))
    assert not all(torch.equal(u, v) for u, v in zip(r[0], r[2]))


def test_unknown_model_is_refused(B):
    with pytest.raises(B.SqsmError) as e:
        B.Context(0).scan_shape([0, 5], model=7)
    assert e.value.code == B.ERR_INVALID_ARG

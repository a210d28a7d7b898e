"""The scan shape that a query reports is the one the calls run with, for every
kind of model, and the default leaf of FP64 coordinated-turn calls."""
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


@pytest.mark.parametrize("n,leaf", [(1, 1), (16_384, 1), (16_385, 2), (65_536, 2), (65_537, 3)])
def test_fp64_coordinated_turn_leaf(B, n, leaf):
    """(these lengths do not depend on the GPU, but 65537 needs 86 SMs)"""
    f64 = torch.float64
    ctx = B.Context(0)
    assert torch.cuda.get_device_properties(0).multi_processor_count >= 86
    for kind in (B.MODEL_CT_BEARINGS, B.MODEL_CT_BEARINGS_R):
        assert ctx.scan_shape([0, n], f64, model=kind) == (leaf, 0)
    y = torch.zeros((n, 2), dtype=f64, device="cuda:0")
    m0 = torch.zeros((1, 5), dtype=f64, device="cuda:0") + 0.1
    N0 = 0.1 * torch.eye(5, dtype=f64, device="cuda:0")[None]
    r = [B.sqsm_ipls_smooth(c, W.CT_THETA_TRUE, y, [0, n], m0, N0, 1, B.EXTENDED)
         for c in (ctx, B.Context(0, leaf_chunk=leaf))]
    torch.cuda.synchronize()
    assert all(torch.equal(u, v) for u, v in zip(*r))


def test_unknown_model_is_refused(B):
    with pytest.raises(B.SqsmError) as e:
        B.Context(0).scan_shape([0, 5], model=7)
    assert e.value.code == B.ERR_INVALID_ARG

"""The log-likelihood's sum over a sequence's leaf chunks in a batch: in slices
or in one launch, by the number of sequences."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2207_00426_gb300 import workloads as W


@pytest.fixture(scope="module")
def B():
    from paper_2207_00426_gb300 import binding
    return binding


def _counts(lengths, dt):
    """Constant counts for a population batch of these lengths."""
    n, nb = sum(lengths), len(lengths)
    return (W.RICKER_THETA_TRUE, torch.full((n, 1), 10.0, dtype=dt, device="cuda:0"),
            np.concatenate([[0], np.cumsum(lengths)]),
            torch.full((nb, 1), W.RICKER_X0, dtype=dt, device="cuda:0"),
            torch.zeros((nb, 1, 1), dtype=dt, device="cuda:0"))


@pytest.mark.parametrize("nb", [63, 64, 65])
@pytest.mark.parametrize("n", [2048, 2049])
def test_long_sequence_in_a_batch(B, n, nb):
    """One step per leaf; `nb` sequences of n chunks (2049: two slices, taken
    for at most 64 sequences) against one alone: the same terms in another
    order, n additions of at most 20 each way."""
    f64 = torch.float64
    ctx = B.Context(0, leaf_chunk=1)
    one = B.sqsm_ipls_smooth_population(ctx, *_counts([n], f64), 2)[2]
    all_ = B.sqsm_ipls_smooth_population(ctx, *_counts([n] * nb, f64), 2)[2]
    torch.cuda.synchronize()
    assert ctx.status() == 0
    assert (all_ - one).abs().max().item() <= 2 * n * 2.0 ** -53 * 20 * n


def test_short_sequences_beside_a_long_one(B):
    """60000 sequences of two steps: a sequence of 1e6 steps beside them adds
    its own sum (a block's 0.13 ms), not a grid of its slices for each."""
    t = {}
    for name, lengths in (("short", [2] * 60_000), ("skewed", [1_000_000] + [2] * 60_000)):
        ctx = B.Context(0)
        ctx.profile(True)
        a = _counts(lengths, torch.float32)
        us = []
        for _ in range(5):
            B.sqsm_ipls_smooth_population(ctx, *a, 1)
            torch.cuda.synchronize()
            us.append(1e3 * ctx.profile_read()["loglik_reduce"][0])
        t[name] = float(np.median(us))
        ctx.close()
    print(t)
    assert t["skewed"] < 4 * t["short"], t

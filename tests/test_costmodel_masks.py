"""The cost model counts the operations that Tria executes with its structural
zeros left out: against the nonzeros that a dense Householder run on a random
matrix of the pattern meets."""
import numpy as np
import pytest

from paper_2207_00426_gb300 import costmodel as CM


def _count(A, nref):
    """Operations of Tria(A) on the entries that are not zero."""
    A, (R, C), f = A.copy(), A.shape, 0
    for i in range(nref):
        x = A[i, i:].copy()
        f += 2 * np.count_nonzero(x) + 6
        v, s = x.copy(), np.linalg.norm(x)
        v[0] += s if x[0] >= 0 else -s
        tau = 2.0 / (v @ v)
        for r in range(i + 1, R):
            both = np.count_nonzero((A[r, i:] != 0) & (v != 0))
            if both:
                f += 2 * both + 1 + 2 * np.count_nonzero(v)
                A[r, i:] -= tau * (A[r, i:] @ v) * v
        A[i, i:] = 0
        A[i, i] = s
        A[i + 1:, i][np.abs(A[i + 1:, i]) < 1e-300] = 0
    return f


@pytest.mark.parametrize("R,C,rows,nref", [
    (5, 10, CM.dense_then_lower(5), 5), (5, 10, CM.few_then_identity(5, 5), 5),
    (5, 10, CM.few_then_identity(2, 5), 5), (5, 10, CM.few_rows_then_identity(2, 5), 5),
    (5, 10, CM.few_then_few_lower(2, 5), 5), (7, 7, CM.dense_lower_over_lower(2, 5), 7),
    (10, 10, CM.dense_lower_over_lower(5, 5), 10), (2, 7, CM.bearing_noise(2, 5), 2),
    (5, 10, None, 5), (6, 12, CM.dense_then_lower(6), 3), (1, 2, CM.dense_then_lower(1), 1)])
def test_tria_counts_the_nonzeros(R, C, rows, nref):
    rng = np.random.default_rng(R * 100 + C)
    A = rng.uniform(0.5, 1.5, (R, C)) * rng.choice([-1, 1], (R, C))
    if rows is not None:
        for i in range(R):
            A[i] *= [rows(i) >> j & 1 for j in range(C)]
    assert CM.tria(R, C, nref, rows) == _count(A, nref)


def test_sizes_of_the_coordinated_turn_model():
    assert CM.tria(5, 10) == 480 and CM.tria(5, 10, rows=CM.dense_then_lower(5)) == 340
    assert CM.tria(5, 10, rows=CM.few_then_identity(5, 5)) == 320
    assert CM.tria(5, 10, rows=CM.few_then_identity(2, 5)) == 186
    assert CM.kf_step(5, 2, masked=True) < CM.kf_step(5, 2)
    assert CM.smoother_element(5, masked=True) == CM.smoother_element(5) - 1535 + 1125
    assert CM.smoother_element(2, masked=True) == CM.smoother_element(2)
    assert CM.filter_combine(5, 2) < CM.filter_combine(5) < 4415   # 4415: every loop dense

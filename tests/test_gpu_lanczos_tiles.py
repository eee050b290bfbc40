"""Lanczos with the tiled fixed-point neighbour sums (n >= 18): one strided pass (n
= 18..21) and two (n = 22, 23), from the uniform and from a random start.

One-literal clauses make H(s) a sum of one-qubit terms, so its levels are sums
of the 2 x 2 matrices' eigenvalues: the ground level takes the lower one of every
qubit, the next level that the uniform start reaches the upper one of the qubit
with the smallest difference among those whose two counts differ.
120 iterations converge both far below the tolerance of the FP64 vectors, n
roundings of 2^-53 of ||H|| per product; the bound allows a thousand times that.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("start", [0, 1], ids=["uniform", "random"])
@pytest.mark.parametrize("n", [17, 18, 19, 20, 21, 22, 23])
def test_one_literal_levels(n, start):
    import paper_1103_1399_gb300 as q
    rng = np.random.default_rng(n)
    s = 0.45
    clauses, lower, upper, seen = [], [], [], []
    for v in range(1, n + 1):
        e = [int(k) for k in rng.integers(0, 4, size=2)]  # violated at x_v = 0 and at x_v = 1
        clauses += [[v]] * e[0] + [[-v]] * e[1]
        h = np.array([[0.5 * (1 - s) + s * e[0], -0.5 * (1 - s)], [-0.5 * (1 - s), 0.5 * (1 - s) + s * e[1]]])
        w = np.linalg.eigvalsh(h)
        lower.append(w[0])
        upper.append(w[1])
        seen.append(e[0] != e[1])  # else the uniform start has no part in the qubit's upper state
    gaps = np.sort((np.array(upper) - np.array(lower))[seen])
    want = [sum(lower), sum(lower) + gaps[0]]
    with q.Instance(n, clauses) as inst:
        got, iters = inst.lowest_eigenvalues(s, k=1 if start else 2, max_iter=120, start=start, seed=7)
    norm = sum(upper)
    assert iters == 120
    for g, w in zip(got, want):
        assert abs(g - w) <= 1000 * n * 2.0**-53 * norm

"""The default plan at n = 31: an 11-bit group whose rows lie within memory pages (layout
H first) and a 10-bit group whose rows lie on pages of their own.  The other order
of 11-bit tiles is that of n = 32 (test_gpu_qbits).  Product instance, angles of both
kinds (one turn per qubit, two turns)."""

import pytest

from test_gpu_qbits import product_check, product_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dt", [(31, 0.1), (31, 4.1), (32, 4.1)])
def test_default_plan(n, dt):
    import torch
    import paper_1103_1399_gb300 as q
    K = 4
    plan, err, o = product_check(q, torch, n, product_instance(n, n), dt * K, K, 3)
    want = ["[10,15)+[15,21)", "[21,26)+[26,31)"] if n == 31 else ["[10,15)+[26,32)", "[15,20)+[20,26)"]
    assert all(w in plan for w in want), plan
    # K steps round an amplitude by a few 2^-24 of itself per turn, phase and fold
    assert err <= K * (2 * n + 8) * 2.0**-24
    assert abs(o["norm"] - 1.0) <= 1e-6

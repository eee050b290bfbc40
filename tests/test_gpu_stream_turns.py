"""One-qubit rotations of the streaming passes in the gauge i^popcount.

Every tile form (groups of 5, 7, 10 and 11 bits) at small angles (one turn per
qubit) and at angles up to 4.1 (two turns where the tangent is above 1 in
magnitude), a run over more steps than one span of the deferred phase, and the
split groups of the default plan beyond L2.
Tolerance: each turn, phase and fold rounds an amplitude by a few 2^-24 of
itself, so K steps leave at most K (2 n + 8) 2^-24 of the unit norm.
"""

import numpy as np
import pytest

import oracle
import satgen
from test_gpu_qbits import product_check, product_instance

pytestmark = pytest.mark.gpu


def passes_run(n, group, dt, K, graph=False):
    import torch
    import paper_1103_1399_gb300 as q
    cl = satgen.random_instance(n, 5 * n, seed=n)
    rng = np.random.default_rng(n)
    psi0 = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi0 = (psi0 / np.linalg.norm(psi0)).astype(np.complex64)
    with q.Instance(n, cl) as inst:
        inst.set_variant(3, group)
        if graph:
            inst.set_launch_mode(q.LAUNCH_GRAPH)
        assert "team" not in inst.describe_plan()
        psi = torch.from_numpy(psi0).cuda()
        inst.evolve(psi, dt * K, K)
    return cl, psi0, psi.cpu().numpy()


@pytest.mark.parametrize("dt", [0.1, 4.1])
@pytest.mark.parametrize("n,group", [(15, 5), (17, 7), (20, 10), (21, 11)])
def test_passes_match_oracle(n, group, dt):
    K = 7
    cl, psi0, got = passes_run(n, group, dt, K)
    ref = oracle.evolve_strang(n, cl, dt * K, K, psi0=psi0.astype(np.complex128))
    assert np.linalg.norm(got.astype(np.complex128) - ref) <= K * (2 * n + 8) * 2.0**-24


@pytest.mark.parametrize("dt", [0.1, 4.1])
def test_long_run_and_its_graph(dt):
    n, K = 15, 1030
    cl, psi0, got = passes_run(n, 5, dt, K)
    assert np.array_equal(got, passes_run(n, 5, dt, K, graph=True)[2])
    ref = oracle.evolve_strang(n, cl, dt * K, K, psi0=psi0.astype(np.complex128))
    assert np.linalg.norm(got.astype(np.complex128) - ref) <= K * (2 * n + 8) * 2.0**-24


@pytest.mark.parametrize("n", [26, 27])
def test_default_split_groups(n):
    import torch
    import paper_1103_1399_gb300 as q
    K = 4
    plan, err, o = product_check(q, torch, n, product_instance(n, n), 0.1 * K, K, 3)
    assert "group bits [10,15)+[%d,%d)" % (n - 5, n) in plan, plan
    assert err <= K * (2 * n + 8) * 2.0**-24
    assert abs(o["norm"] - 1.0) <= 1e-6

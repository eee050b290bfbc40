"""One-qubit rotations in the gauge i^popcount (the sizes whose state stays on
chip, n <= 21): every register window, lane layout and CTA team, at angles of
both row forms, and runs longer than one launch.

Steps of dt = 4.1 take theta = dt (1 - s) over (0, 4.1): tan(theta/2) below and
above 1 in magnitude and cos(theta/2) of both signs, from a random state and
over a sub-range, so that odd and even step counts end in either layout.
Tolerance: each turn, phase and fold rounds an amplitude by a few 2^-24 of
itself, so K steps leave at most K (2 n + 8) 2^-24 of the unit norm.
"""

import numpy as np
import pytest

import oracle
import satgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K", [(n, K) for n in range(1, 22) for K in (7, 18)] + [(8, 1030), (13, 1030), (15, 1030)])
def test_large_angles_match_oracle(n, K):
    import torch
    import paper_1103_1399_gb300 as q
    cl = satgen.random_instance(n, 5 * n, seed=n, width=min(3, n))
    rng = np.random.default_rng(n)
    psi0 = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi0 = (psi0 / np.linalg.norm(psi0)).astype(np.complex64)
    T = 4.1 * K
    ref = oracle.evolve_strang(n, cl, T, K, psi0=psi0.astype(np.complex128))
    with q.Instance(n, cl) as inst:
        psi = torch.from_numpy(psi0).cuda()
        inst.evolve(psi, T, K)
    assert np.linalg.norm(psi.cpu().numpy().astype(np.complex128) - ref) <= K * (2 * n + 8) * 2.0**-24

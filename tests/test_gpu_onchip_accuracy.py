"""Rounding of the evolvers that keep the state on chip, by what it does to the observables.

Late in a sweep a few amplitudes carry <H_P> and the ground probability, and a
random walk of their roundings is the error of both.  One rounding of an
amplitude per step, uniform within 2^-24 of it, leaves about sqrt(K / 6) 2^-24 =
4.9e-7 of the amplitude after K = 400 steps; four leave twice that.  The evolvers
carry what a rounding leaves out, so the bar is half of the single rounding's
figure, on the root mean square over the instances (relative errors against the
complex128 oracle).  The state's own error also holds what the rounded angles and
phase rows leave, up to 2^-24 of a turn each: the single rounding's figure.
"""

import numpy as np
import pytest

import oracle
import satgen

pytestmark = pytest.mark.gpu

K = 400
ONE = (K / 6) ** 0.5 * 2.0**-24


@pytest.mark.parametrize("n,seeds", [(8, 8), (11, 8), (12, 8), (14, 4), (16, 4)])
def test_observables_over_400_steps(n, seeds):
    import torch
    import paper_1103_1399_gb300 as q
    T = 0.05 * K
    errs = []
    for seed in range(seeds):
        cl = satgen.planted_instance(n, 100 * n + seed)["clauses"]
        E = oracle.violated_counts(n, cl)
        ref = oracle.evolve_strang(n, cl, T, K)
        p = np.abs(ref) ** 2
        low = E == 0
        with q.Instance(n, cl) as inst:
            psi = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
            inst.init_uniform(psi)
            inst.evolve(psi, T, K)
            hp = inst.observables(psi)["expect_hp"]
            got = psi.cpu().numpy().astype(np.complex128)
        want_hp, want_low = float((p * E).sum()), float(p[low].sum())
        errs.append([np.linalg.norm(got - ref), hp / want_hp - 1, float((np.abs(got[low]) ** 2).sum()) / want_low - 1])
    rms = np.sqrt((np.array(errs) ** 2).mean(axis=0))
    assert rms[0] <= ONE and rms[1] <= ONE / 2 and rms[2] <= ONE / 2, rms


@pytest.mark.parametrize("n", [11, 13, 16, 19])
def test_steps_of_very_different_angles(n):
    """Angles between none and two turns of a quarter circle, in any order: the scales of
    neighbouring steps differ by up to 2^n."""
    import torch
    import paper_1103_1399_gb300 as q
    cl = satgen.random_instance(n, 5 * n, seed=n)
    rng = np.random.default_rng(n)
    steps = 40
    s = rng.choice([0.0, 0.5, 0.99, 1.0], size=steps)
    dt = 3.0
    psi0 = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi0 = (psi0 / np.linalg.norm(psi0)).astype(np.complex64)
    ref = oracle.evolve_strang(n, cl, dt * steps, steps, psi0=psi0.astype(np.complex128), s_values=s)
    with q.Instance(n, cl) as inst:
        psi = torch.from_numpy(psi0).cuda()
        inst.evolve_schedule(psi, dt, s)
    err = np.linalg.norm(psi.cpu().numpy().astype(np.complex128) - ref)
    # every turn, phase and fold rounds at random: sqrt of the worst case's count
    assert err <= (steps * (2 * n + 8)) ** 0.5 * 2.0**-24 * 2, err

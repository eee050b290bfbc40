"""An explicit variant runs the streaming passes, also where the default is a team of
CTAs (15 <= n <= 21), with and without a group width and after an autotuned plan.

Tolerance: as for the passes with a group width (test_gpu_stream_turns).
"""

import numpy as np
import pytest

import oracle
import satgen

pytestmark = pytest.mark.gpu

K, DT = 7, 0.1


def launches(inst, psi):
    inst.profile(True)
    inst.profile_reset()
    inst.evolve(psi, DT * K, K)
    out = {k: v[0] for k, v in inst.profile_read().items()}
    inst.profile(False)
    return out


@pytest.mark.parametrize("n,group", [(15, 0), (18, 0), (20, 0), (21, 0), (21, 11)])
def test_rotation_variant_runs_the_passes(n, group):
    import torch
    import paper_1103_1399_gb300 as q
    cl = satgen.random_instance(n, 5 * n, seed=n)
    ref = oracle.evolve_strang(n, cl, DT * K, K)
    with q.Instance(n, cl) as inst:
        assert "team" in inst.describe_plan()
        inst.set_variant(3, group)
        assert "team" not in inst.describe_plan()
        psi = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
        inst.init_uniform(psi)
        ran = launches(inst, psi)
        assert ran["onchip"] == 0 and ran["low_merge"] + ran["low_last"] + ran["low_first"] == K + 1, ran
    assert np.linalg.norm(psi.cpu().numpy().astype(np.complex128) - ref) <= K * (2 * n + 8) * 2.0**-24


def test_rotation_variant_runs_the_passes_after_tuning():
    import torch
    import paper_1103_1399_gb300 as q
    n = 16
    cl = satgen.random_instance(n, 5 * n, seed=n)
    try:
        with q.Instance(n, cl) as inst:
            psi = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
            inst.autotune(psi, steps=2)
        with q.Instance(n, cl) as inst:
            inst.set_variant(3)
            assert "team" not in inst.describe_plan()
            inst.init_uniform(psi)
            assert launches(inst, psi)["onchip"] == 0
    finally:
        q.forget_tuned_plans()

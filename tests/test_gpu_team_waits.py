"""The team evolver's bounded waits (cluster, word and grid-barrier exchange).

An injected fault makes one CTA withhold its first exchange: every other CTA's
wait runs out, the kernel returns, the next synchronising call reports
QAA_E_TIMEOUT once, and the same handle then evolves as a fresh one does, bit
for bit.
"""

import pytest

import satgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [12, 14, 15, 18, 20, 21])
def test_lost_exchange_times_out_and_the_handle_recovers(n):
    import torch
    import paper_1103_1399_gb300 as q
    cl = satgen.planted_instance(n, 3 * n)["clauses"]
    T, K = 1.0, 20

    def evolved(inst):
        psi = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
        inst.init_uniform(psi)
        inst.evolve(psi, T, K)
        return psi

    with q.Instance(n, cl) as fresh:
        want = evolved(fresh)
        fresh.observables(want)
    with q.Instance(n, cl) as inst:
        inst.inject(1)
        psi = evolved(inst)
        with pytest.raises(q.QaaError) as ei:
            inst.observables(psi)
        assert ei.value.status == -4
        got = evolved(inst)
        assert abs(inst.observables(got)["norm"] - 1.0) <= 1e-6
        assert torch.equal(got, want)


def test_faults_that_cannot_be_injected_are_refused():
    import paper_1103_1399_gb300 as q
    with q.Instance(8, [[1, 2, 3]]) as inst:
        with pytest.raises(q.QaaError):
            inst.inject(1)
        with pytest.raises(q.QaaError):
            inst.inject(7)

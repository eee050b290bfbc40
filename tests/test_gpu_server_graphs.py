"""Launch graphs of the server's streamed requests, at sizes that run as passes by default
(n >= 22; smaller ones run on a team of CTAs, which needs no graph).

The request's memory block shows which form was chosen: a launch graph keeps
phase rows of nine steps, per-pass launches those of the whole (short) run.
"""

import pytest

import satgen
from test_gpu_serving import wait_all

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,T,K", [(22, 3.0, 40), (23, 4.0, 19)])
def test_graph_requests_equal_per_pass_requests(n, T, K, monkeypatch):
    import paper_1103_1399_gb300 as q
    cl = satgen.planted_instance(n, 31)["clauses"]

    def serve():
        with q.Server(max_slots=2) as srv:
            res = wait_all(srv, [srv.submit(n, cl, T, K)])
            return next(iter(res.values())), srv.stats()["peak_used_bytes"]

    monkeypatch.delenv("QAA_SERVER_GRAPH_BITS", raising=False)
    passes, passes_bytes = serve()
    monkeypatch.setenv("QAA_SERVER_GRAPH_BITS", "23")
    graph, graph_bytes = serve()
    assert graph_bytes < passes_bytes
    assert passes["status"] == graph["status"] == 0
    for k in ("success_prob", "norm", "energy", "expect_hb", "ground_count"):
        assert passes[k] == graph[k], (k, passes, graph)

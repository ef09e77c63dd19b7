"""The executable graphs that fmg_solve_uneven keeps: batches whose numbers of
samples lie on both sides of the line where FP64 smoothing changes its launches
have different graphs, both of which stay."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("converged", [0, 1])
def test_alternating_counts_instantiate_once_each(converged):
    import paper_1910_04727_gb300 as fm
    c = fm.Context(1, 128, 8, converged=converged, tol=1e-8, max_cycles=50)
    K = torch.tensor(W.smooth_lognormal_field(128, S=4, tag=5200), device="cuda").repeat(35, 1, 1)
    few, many = [K[:3].contiguous()], [K.contiguous()]   # 48 Ki and 2.2 Mi cells
    want = {id(g): c.fmg_solve_batch(g[0])[:2] for g in (few, many)}
    for _ in range(3):
        for g in (few, many):
            (qf, qc, _), = c.solve_uneven(g)
            assert torch.equal(qf, want[id(g)][0]) and torch.equal(qc, want[id(g)][1])
    assert c.uneven_stats() == dict(instantiations=2, updates=4, launches=6)


def test_calls_with_and_without_the_status_keep_a_graph_each():
    import paper_1910_04727_gb300 as fm
    c = fm.Context(1, 128, 8, converged=1, tol=1e-8, max_cycles=50)
    K = [torch.tensor(W.smooth_lognormal_field(128, S=3, tag=5201), device="cuda")]
    for want in (True, False) * 3:
        c.solve_uneven(K, want_status=want)
    assert c.uneven_stats() == dict(instantiations=2, updates=4, launches=6)

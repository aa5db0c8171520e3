"""A planned mesh takes no more device memory than a server charges its budget for it
(serve.cu: 48 planes, 3 + 2 records and two row lists per vertex, edges, tables)."""
import numpy as np
import pytest

from paper_1604_06525_gb300 import synth

pytestmark = pytest.mark.gpu


def charged(V, E, n_handles):
    pl = (V + 31) // 32 * 32
    return 68 * pl * 4 + 16 * E + 8 * pl + 16 * n_handles + (1 << 16)


def chain(V):
    """Two edges a vertex: the records, not the edges, are what it takes."""
    rng = np.random.default_rng(V)
    U = np.stack([np.arange(V), np.zeros(V), np.zeros(V)]).astype(np.float32)
    a, b = np.arange(V - 1, dtype=np.int32), np.arange(1, V, dtype=np.int32)
    return synth.MeshProblem(V, U, np.concatenate([a, b]), np.concatenate([b, a]),
                             np.zeros((6, V), np.float32), np.array([0, V - 1], np.int32),
                             rng.standard_normal((2, 3)).astype(np.float32), 1.0, 10.0)


@pytest.mark.parametrize("case", ["tiny", "small", "chain", "mesh"])
def test_planned_meshes_fit_their_estimate(case):
    import ctypes
    from paper_1604_06525_gb300 import api
    prob = {"tiny": lambda: chain(4), "small": lambda: synth.mesh_problem(1, seed=1, handle_frac=0.05),
            "chain": lambda: chain(60000), "mesh": lambda: synth.mesh_problem(5, seed=1)}[case]()
    g = api.Problem(prob)
    used = ctypes.c_size_t()
    assert g.lib.opt_selftest_footprint(g.h, ctypes.byref(used)) == 0
    assert used.value <= charged(prob.V, prob.v0.size, prob.handle_idx.size)
    g.close()


def test_request_without_memory_beside_others_is_planned_alone():
    import torch
    from paper_1604_06525_gb300 import api
    srv = api.Server(1 << 30, outer=2, inner=4, rel_tol=0.0)
    tickets = [srv.submit(synth.warp_problem(40 + 9 * i, 33, 6, seed=i)) for i in range(4)]
    tickets.append(srv.submit(synth.mesh_problem(2, seed=1, handle_frac=0.05)))
    srv.lib.opt_selftest_refuse_allocation()              # one of the plans finds no memory
    busy = True
    while busy:
        active, queued = srv.step()
        busy = active + queued > 0
    for t in tickets:
        report, x = srv.poll(t)
        assert report["outer_done"] == 2 and torch.isfinite(x).all()
    srv.close()

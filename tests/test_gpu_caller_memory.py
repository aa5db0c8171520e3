"""Caller planes at any address: the unknowns of a grid or of the float64 solver may
start at a byte offset that a kernel cannot address element by element.  The same
bits come back as from aligned planes."""
import ctypes

import numpy as np
import pytest

from paper_1604_06525_gb300 import synth

pytestmark = pytest.mark.gpu


def shifted(x, offset):
    """A copy of x (planes first) in raw memory, `offset` bytes behind an aligned
    address; returns the storage, the planes' addresses and a reader."""
    import torch
    n, bytes_ = x.shape[0], x[0].numel() * x.element_size()
    room = (bytes_ + 255) // 256 * 256 + 256
    raw = torch.zeros(n * room, dtype=torch.uint8, device="cuda")
    cut = [raw[c * room + offset:c * room + offset + bytes_] for c in range(n)]
    for c in range(n):
        cut[c].copy_(x[c].reshape(-1).view(torch.uint8))
    return raw, [c.data_ptr() for c in cut], lambda: np.stack([c.cpu().numpy().view(x.cpu().numpy().dtype) for c in cut])


@pytest.mark.parametrize("offset", [1, 2, 4])
@pytest.mark.parametrize("kind", ["warp", "poisson", "warp64", "mesh64"])
@pytest.mark.parametrize("method,graph", [("gn", 1), ("lm", 0)])
def test_unaligned_unknowns_solve_like_aligned_ones(kind, offset, method, graph):
    import torch
    from paper_1604_06525_gb300 import api
    prob = (synth.warp_problem(60, 21, 7, seed=3) if kind.startswith("warp") else
            synth.poisson_problem(52, 33, seed=4) if kind == "poisson" else synth.mesh_problem(2, seed=5, handle_frac=0.05))
    f64 = kind.endswith("64")
    plain = (api.ProblemF64 if f64 else api.Problem)(prob)
    lib = plain.lib
    desc, x, keep = (api.make_descriptor_f64 if f64 else api.make_descriptor)(prob, "cuda")
    raw, ptrs, read = shifted(x, offset)
    for c, p in enumerate(ptrs):
        desc.unknowns[c] = p
    name = ("grid" if not kind.startswith("mesh") else "graph") + ("_f64" if f64 else "")
    h = ctypes.c_void_p()
    assert getattr(lib, "opt_problem_create_" + name)(ctypes.byref(desc), None, ctypes.byref(h)) == 0
    try:
        want = getattr(plain, "solve_" + method)(2, 4, use_graph=graph)
        p = api.default_params(outer=2, inner=4, use_graph=graph, stream=torch.cuda.current_stream().cuda_stream)
        hist = (ctypes.c_double * 3)()
        rep = api.Report()
        rep.E_history = ctypes.cast(hist, ctypes.POINTER(ctypes.c_double))
        solve = getattr(lib, "opt_solve_" + method + ("_f64" if f64 else ""))
        assert solve(h, ctypes.byref(p), ctypes.byref(rep)) == 0
        assert list(hist[:rep.outer_done + 1]) == want["E_history"]
        np.testing.assert_array_equal(read(), plain.x.cpu().numpy().reshape(x.shape[0], -1))
    finally:
        getattr(lib, "opt_problem_destroy" + ("_f64" if f64 else ""))(h)
    plain.close()

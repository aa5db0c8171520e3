"""The routes of a solve that differ in where the work runs, not in what it computes.

* A solve of one problem keeps the PCG state on chip where it fits (resident loop: one
  cluster for small problems, else the whole device); a batch takes one launch per
  phase.  A row is the same arithmetic in the same order on both, and the sums are
  compensated, so a difference can only come from a rounding of alpha or beta
  (6e-8 each): 14 iterations stay below TOL.
* The grid energies read the planes quad by quad; against the float64 oracle.
* The float64 solver runs its loop in one launch; against the oracle.
* The server plans several requests at once; a bad one fails alone.
"""
import numpy as np
import pytest

import oracle
from paper_1604_06525_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 2e-6
TOL_ENERGY = 1e-5          # float32 residuals, compensated sums
TOL_F64 = 1e-9


def one_way(prob, keep, seed):
    """A random part of the directed edges, a few of them twice."""
    rng = np.random.default_rng(seed)
    sel = rng.random(prob.v0.size) < keep
    v0, v1 = prob.v0[sel], prob.v1[sel]
    dup = rng.choice(v0.size, size=5, replace=False)
    v0, v1 = np.concatenate([v0, v0[dup]]), np.concatenate([v1, v1[dup]])
    order = np.lexsort((v1, v0))
    prob.v0, prob.v1 = v0[order].astype(np.int32), v1[order].astype(np.int32)
    return prob


def make(case):
    kind, *a = case
    if kind == "warp":
        W, H, masked = a
        mask = synth.random_mask(W, H, 0.2, seed=W) if masked else None
        return synth.warp_problem(W, H, max(1, W * H // 300), seed=W + H, max_disp=2.0, mask=mask)
    if kind == "poisson":
        return synth.poisson_problem(a[0], a[1], seed=a[0])
    if kind in ("cutout", "patch"):        # whole cells and tiles without an unknown
        W, H = a
        mask = np.ones((H, W), np.uint8)
        mask[H // 3:H // 3 + 11, 5:W - 3] = 0
        mask[:, W // 2] = 0
        if kind == "patch":
            return synth.poisson_problem(W, H, seed=4, mask=mask)
        return synth.warp_problem(W, H, 9, seed=6, max_disp=2.0, mask=mask)
    if kind == "graph":
        return synth.warp_graph_from_grid(make(("warp", *a)))
    if kind == "volume":
        return synth.volume_problem(*a, max(1, a[0] * a[1] * a[2] // 90), seed=sum(a), max_off=0.4)
    if kind == "embedded":
        return synth.embedded_problem(a[0], seed=7, handle_frac=0.05)
    prob = synth.mesh_problem(a[0], seed=9, handle_frac=0.05)
    return one_way(prob, a[1], 3) if a[1] < 1.0 else prob


# sizes around the edges of the routes: one block, one cluster (up to 8,192 units), the
# device; ragged tiles and runs, odd quads, masks, one-way edges
CASES = [("warp", 1, 1, 0), ("warp", 37, 5, 0), ("warp", 64, 64, 1), ("warp", 127, 65, 0), ("warp", 300, 57, 1),
         ("warp", 411, 303, 0), ("poisson", 37, 29), ("poisson", 130, 63), ("poisson", 500, 333),
         ("cutout", 200, 90), ("cutout", 37, 61), ("patch", 301, 77), ("patch", 40, 200),
         ("graph", 33, 17, 1), ("graph", 111, 99, 0), ("volume", 5, 4, 3), ("volume", 31, 21, 13),
         ("embedded", 1), ("embedded", 4), ("mesh", 0, 1.0), ("mesh", 3, 0.6), ("mesh", 5, 1.0), ("mesh", 6, 0.7)]


@pytest.mark.parametrize("method", ["gn", "lm"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_solo_solve_equals_batch(case, method):
    import torch
    from paper_1604_06525_gb300 import api
    prob = make(case)
    solo = api.Problem(prob)
    r = (solo.solve_gn if method == "gn" else solo.solve_lm)(2, 7)
    member = api.Problem(prob)
    batch = api.Batch([member])
    (b,), _ = (batch.solve_gn if method == "gn" else batch.solve_lm)(2, 7)
    torch.cuda.synchronize()
    x, y = solo.x.cpu().numpy().astype(np.float64), member.x.cpu().numpy().astype(np.float64)
    batch.close()
    assert np.isfinite(x).all()
    assert r["pcg_done"] == b["pcg_done"] and r["accepted"] == b["accepted"]
    assert np.linalg.norm(x - y) <= TOL * max(np.linalg.norm(y), 1e-30)
    for s, t in zip(r["E_history"], b["E_history"]):
        assert abs(s - t) <= 1e-5 * max(abs(t), 1e-3 * abs(b["E_history"][0]))


@pytest.mark.parametrize("W,H,masked", [(1, 1, 0), (3, 9, 0), (32, 8, 1), (33, 9, 1), (128, 8, 0), (131, 17, 1),
                                        (260, 40, 0)])
@pytest.mark.parametrize("kind", ["warp", "poisson"])
def test_grid_energies_match_oracle(kind, W, H, masked):
    from paper_1604_06525_gb300 import api
    mask = synth.random_mask(W, H, 0.3, seed=3) if masked else None
    if kind == "warp":
        prob = synth.warp_problem(W, H, max(1, W * H // 40), seed=W, max_disp=2.0, mask=mask, x0_noise=0.4)
    else:
        prob = synth.poisson_problem(W, H, seed=W, mask=mask)
    e = oracle.make_energy(prob)
    g = api.Problem(prob)
    ref = oracle.jtf_diag(e, prob.x0.reshape(-1).astype(np.float64))[2]
    assert abs(g.energy() - ref) <= TOL_ENERGY * max(abs(ref), 1e-12)
    # a trial energy and its model value decide the first LM step as the oracle does
    r = g.solve_lm(1, 3)
    want = oracle.levenberg_marquardt(e, prob.x0.reshape(-1), 1, 3)
    # (an energy far below the first one is a difference of near equals in float32)
    assert abs(r["E_final"] - want.E_history[-1]) <= 1e-4 * max(abs(want.E_history[-1]), 1e-2 * ref)
    g.close()


@pytest.mark.parametrize("method", ["gn", "lm"])
@pytest.mark.parametrize("case", [("warp", 1, 1, 0), ("warp", 41, 23, 1), ("poisson", 45, 31), ("mesh", 0, 1.0),
                                  ("mesh", 2, 0.6), ("mesh", 4, 1.0)], ids=lambda c: "-".join(map(str, c)))
def test_float64_loop_matches_oracle(case, method):
    from paper_1604_06525_gb300 import api
    prob = make(case)
    e = oracle.make_energy(prob)
    g = api.ProblemF64(prob)
    r = (g.solve_gn if method == "gn" else g.solve_lm)(2, 6)
    f = oracle.gauss_newton if method == "gn" else oracle.levenberg_marquardt
    want = f(e, prob.x0.reshape(-1).astype(np.float64), 2, 6)
    for s, t in zip(r["E_history"], want.E_history):
        assert abs(s - t) <= TOL_F64 * max(abs(t), 1e-6 * abs(want.E_history[0]))
    g.close()


def test_requests_planned_together_fail_alone():
    import torch
    from paper_1604_06525_gb300 import api
    probs = [synth.warp_problem(40 + 9 * i, 33, 6, seed=i) for i in range(5)]
    probs += [synth.mesh_problem(2, seed=20 + i, handle_frac=0.05) for i in range(3)]
    bad = synth.mesh_problem(2, seed=30, handle_frac=0.05)
    bad.v1 = bad.v1.copy()
    bad.v1[5] = bad.V + 3                                    # an edge to nowhere
    srv = api.Server(1 << 30, outer=3, inner=6, rel_tol=0.0)
    tickets = [srv.submit(p) for p in probs[:4] + [bad] + probs[4:]]
    busy = True
    while busy:
        active, queued = srv.step()
        busy = active + queued > 0
    for k, t in enumerate(tickets):
        if k == 4:
            with pytest.raises(api.OptError):
                srv.poll(t)
            continue
        report, x = srv.poll(t)
        alone = api.Problem(probs[k if k < 4 else k - 1])
        want = alone.solve_lm(3, 6)
        assert report["accepted"] == want["accepted"]
        y = alone.x.cpu().numpy().astype(np.float64)
        got = x.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(got - y) <= TOL * np.linalg.norm(y)
        alone.close()
    torch.cuda.synchronize()
    srv.close()


@pytest.mark.parametrize("kind", ["warp", "mesh", "mesh64"])
def test_repeated_solves_equal_fresh_ones(kind):
    """Nothing of a call (its method, preconditioner, history length, a product in
    between) stays in the next one's descriptor, graph or results."""
    from paper_1604_06525_gb300 import api
    prob = make(("warp", 150, 40, 1)) if kind == "warp" else make(("mesh", 3, 1.0))
    cls = api.ProblemF64 if kind.endswith("64") else api.Problem
    calls = [("gn", 2, 5, {}), ("lm", 3, 4, {}), ("lm", 3, 4, {}), ("gn", 5, 3, {"use_precond": 0}), ("gn", 2, 5, {}),
             ("lm", 2, 6, {"use_graph": 0}), ("lm", 6, 2, {})]
    g = cls(prob)
    x0 = g.x.clone()
    batch_members = [] if kind.endswith("64") else [api.Problem(prob), api.Problem(prob)]
    batch = api.Batch(batch_members) if batch_members else None
    for method, outer, inner, kw in calls:
        fresh = cls(prob)
        want = getattr(fresh, "solve_" + method)(outer, inner, **kw)
        g.x.copy_(x0)
        got = getattr(g, "solve_" + method)(outer, inner, **kw)
        assert got["E_history"] == want["E_history"] and got["pcg_done"] == want["pcg_done"]
        np.testing.assert_array_equal(g.x.cpu().numpy(), fresh.x.cpu().numpy())
        fresh.close()
        g.eval_jtf()
        if batch:
            for m in batch_members:
                m.x.copy_(x0)
            reports, _ = getattr(batch, "solve_" + method)(outer, inner, **kw)
            for r in reports:
                assert len(r["E_history"]) == len(want["E_history"])
                for s, t in zip(r["E_history"], want["E_history"]):
                    assert abs(s - t) <= 1e-5 * max(abs(t), 1e-3 * abs(want["E_history"][0]))
    if batch:
        batch.close()
    g.close()


@pytest.mark.parametrize("V,degree", [(2, 1), (60, 46), (60, 47), (60, 48), (60, 49), (9000, 3000)])
def test_planned_edges_match_oracle(V, degree):
    """Edges in any order, both ways or one way, some twice, a hub row around the length
    where the row sort changes its method, and vertices without an edge."""
    import torch
    from paper_1604_06525_gb300 import api
    rng = np.random.default_rng(V + degree)
    hub = rng.choice(np.arange(1, V), size=degree, replace=False)
    a = np.concatenate([np.zeros(degree, int), rng.integers(0, V // 2 + 1, V)])
    b = np.concatenate([hub, rng.integers(0, V // 2 + 1, V)])
    keep = a != b
    a, b = a[keep], b[keep]
    back = rng.random(a.size) < 0.7
    v0, v1 = np.concatenate([a, b[back], a[:3]]), np.concatenate([b, a[back], b[:3]])
    order = rng.permutation(v0.size)
    prob = synth.MeshProblem(V, rng.standard_normal((3, V)).astype(np.float32), v0[order].astype(np.int32),
                             v1[order].astype(np.int32), 0.2 * rng.standard_normal((6, V)).astype(np.float32),
                             np.array([0, V - 1], np.int32), rng.standard_normal((2, 3)).astype(np.float32),
                             0.3, 7.0)                       # (weights whose sums round)
    e = oracle.make_energy(prob)
    x = prob.x0.reshape(-1).astype(np.float64)
    g = api.Problem(prob)
    p = rng.standard_normal(6 * V).astype(np.float32)
    q, _ = g.apply_jtj(torch.as_tensor(p, device="cuda"), 0.0)
    _, diag, E = oracle.jtf_diag(e, x)
    want = oracle.apply_jtj(e, x, p.astype(np.float64), 0.0, np.clip(diag, 1e-6, 1e32))
    assert np.linalg.norm(q.cpu().numpy().reshape(-1) - want) <= 1e-5 * np.linalg.norm(want)
    _, d, Eg = g.eval_jtf()
    np.testing.assert_allclose(d.cpu().numpy().reshape(-1), diag, rtol=2e-4, atol=1e-6)
    assert abs(Eg - E) <= 1e-5 * abs(E)
    g.close()

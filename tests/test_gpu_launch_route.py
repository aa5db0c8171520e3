"""The PCG loop in launches (persistent = -1, and what does not fit on chip) beside the
loop on chip: the launch kernels inside a solve against the oracle, both routes against
each other, several solves at once, and the device-wide loop solve after solve.

Tolerances: rows are the same arithmetic on both routes and every sum is compensated, so
x differs by roundings of alpha and beta (6e-8 each; 14 iterations stay below TOL); the
tiled apply rounds a row in another order, which energies show at 1e-6 (as in
test_gpu_parity.py); float64 against the oracle 1e-9 of the first energy."""
import threading

import numpy as np
import pytest

import oracle
from paper_1604_06525_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 2e-6
TOL_ENERGY = 1e-4
TOL_F64 = 1e-9


def make(kind):
    if kind == "warp_small":
        return synth.warp_problem(61, 40, 9, seed=3, max_disp=2.0)
    if kind == "warp":
        return synth.warp_problem(150, 141, 20, seed=2, max_disp=2.0, mask=synth.random_mask(150, 141, 0.2, seed=1))
    if kind == "poisson":
        return synth.poisson_problem(300, 200, seed=2)
    if kind == "graph":
        return synth.warp_graph_from_grid(synth.warp_problem(40, 31, 9, seed=4, max_disp=2.0))
    if kind == "volume":
        return synth.volume_problem(13, 9, 8, 12, seed=6, max_off=0.4)
    if kind == "embedded":
        return synth.embedded_problem(3, seed=7, handle_frac=0.05)
    return synth.mesh_problem(3 if kind == "mesh_small" else 5, seed=9, handle_frac=0.05)


KINDS = ["warp_small", "warp", "poisson", "graph", "volume", "embedded", "mesh_small", "mesh"]


def energies_match(got, want, tol, floor=0.0):
    assert len(got) == len(want)
    for a, b in zip(got, want):
        assert abs(a - b) <= tol * max(abs(b), floor * abs(want[0]))


@pytest.mark.parametrize("method", ["gn", "lm"])
@pytest.mark.parametrize("kind", KINDS)
def test_launches_match_the_loop_and_the_oracle(kind, method):
    from paper_1604_06525_gb300 import api
    prob = make(kind)
    on_chip, g = api.Problem(prob), api.Problem(prob)
    a = getattr(on_chip, "solve_" + method)(2, 7)
    b = getattr(g, "solve_" + method)(2, 7, persistent=-1)
    assert g.lib.opt_selftest_lose_block(g.h) == 1               # nothing was set up for the loop
    assert a["pcg_done"] == b["pcg_done"] and a["accepted"] == b["accepted"]
    x, y = (p.x.cpu().numpy().astype(np.float64) for p in (on_chip, g))
    assert np.linalg.norm(x - y) <= TOL * np.linalg.norm(y)
    f = oracle.gauss_newton if method == "gn" else oracle.levenberg_marquardt
    ref = f(oracle.make_energy(prob), prob.x0.reshape(-1).astype(np.float64), 2, 7)
    energies_match(b["E_history"], ref.E_history, TOL_ENERGY, 1e-3)
    on_chip.close()
    g.close()


@pytest.mark.parametrize("kind", ["warp_small", "warp", "poisson", "mesh"])
def test_granularities_of_the_launches_agree(kind):
    import torch
    from paper_1604_06525_gb300 import api
    prob = make(kind)
    g = api.Problem(prob)
    ref = g.solve_lm(2, 7, persistent=-1)
    for per in (-1, -8, 1, 4, 64):
        g.set_chunking(per)
        g.x.copy_(torch.as_tensor(prob.x0, device="cuda").reshape(g.x.shape))
        energies_match(g.solve_lm(2, 7, persistent=-1)["E_history"], ref["E_history"], 1e-6, 1e-3)
    g.close()


@pytest.mark.parametrize("route", ["solo", "batch"])
@pytest.mark.parametrize("level", [2, 4])
def test_tiled_apply_inside_a_solve(level, route):
    """k_mesh_apply_tiled with the direction formed in the tile and its halo."""
    from paper_1604_06525_gb300 import api
    prob = synth.mesh_problem(level, seed=12, handle_frac=0.05)
    ref = oracle.levenberg_marquardt(oracle.make_energy(prob), prob.x0.reshape(-1).astype(np.float64), 3, 8)
    runs = []
    for form in (1, 0):
        members = [api.Problem(prob) for _ in range(1 if route == "solo" else 2)]
        for m in members:
            m.set_apply_form(form)
        if route == "solo":
            runs.append(members[0].solve_lm(3, 8, persistent=-1))
        else:
            batch = api.Batch(members)
            reports, _ = batch.solve_lm(3, 8)
            assert reports[0]["E_history"] == reports[1]["E_history"]
            runs.append(reports[0])
            batch.close()
        energies_match(runs[-1]["E_history"], ref.E_history, TOL_ENERGY, 1e-3)
        for m in members:
            m.close()
    energies_match(runs[0]["E_history"], runs[1]["E_history"], 1e-6, 1e-3)


@pytest.mark.parametrize("method", ["gn", "lm"])
@pytest.mark.parametrize("kind", ["warp_small", "poisson_small", "mesh_small"])
def test_float64_launches_match_oracle(kind, method):
    import torch
    from paper_1604_06525_gb300 import api
    prob = synth.poisson_problem(70, 41, seed=5) if kind == "poisson_small" else make(kind)
    g = api.ProblemF64(prob)
    r = getattr(g, "solve_" + method)(2, 6, persistent=-1)
    f = oracle.gauss_newton if method == "gn" else oracle.levenberg_marquardt
    want = f(oracle.make_energy(prob), prob.x0.reshape(-1).astype(np.float64), 2, 6)
    energies_match(r["E_history"], want.E_history, TOL_F64, 1.0)
    # the same handle on chip, and back: the graph of one route is not replayed for the other
    for persistent in (0, -1):
        g.x.copy_(torch.as_tensor(prob.x0.astype(np.float64), device="cuda").reshape(g.x.shape))
        s = getattr(g, "solve_" + method)(2, 6, persistent=persistent)
        energies_match(s["E_history"], want.E_history, TOL_F64, 1.0)
    assert s["E_history"] == r["E_history"]
    g.close()


# the largest states the float64 loop takes (several elements a thread) and the next ones up
@pytest.mark.parametrize("kind,n,fits", [("poisson", 510, True), ("poisson", 530, False), ("warp", 590, True),
                                         ("warp", 610, False), ("mesh", 7, True)])
def test_float64_routes_at_the_loops_capacity(kind, n, fits):
    from paper_1604_06525_gb300 import api
    prob = (synth.poisson_problem(n, n, seed=1, mask=np.zeros((n, n), np.uint8)) if kind == "poisson" else
            synth.warp_problem(n, n, 60, seed=1) if kind == "warp" else synth.mesh_problem(n, seed=1))
    a, b = api.ProblemF64(prob), api.ProblemF64(prob)
    assert (a.lib.opt_selftest_lose_block_f64(a.h) == 0) == fits
    if fits:
        with pytest.raises(api.OptError):
            a.solve_lm(1, 2)                              # (the block it lost)
        a.x.copy_(b.x)
    ra, rb = a.solve_lm(2, 8), b.solve_lm(2, 8, persistent=-1)
    energies_match(ra["E_history"], rb["E_history"], TOL_F64, 1.0)
    x, y = a.x.cpu().numpy(), b.x.cpu().numpy()
    assert np.linalg.norm(x - y) <= TOL_F64 * np.linalg.norm(y)
    a.close()
    b.close()


@pytest.mark.parametrize("persistent", [0, -1])
def test_solves_on_streams_of_their_own(persistent):
    """Several problems at once, each from its own thread on its own stream, among them
    loops over the whole device: the bits of solves one after the other."""
    import torch
    from paper_1604_06525_gb300 import api
    probs = [make(k) for k in ("warp", "poisson", "mesh", "warp_small")]
    want = []
    for p in probs:
        g = api.Problem(p)
        r = g.solve_lm(3, 9, persistent=persistent)
        want.append((r["E_history"], g.x.cpu().numpy()))
        g.close()
    f64 = api.ProblemF64(make("mesh_small"))
    want64 = f64.solve_lm(3, 9, persistent=persistent)["E_history"]
    x64 = torch.as_tensor(make("mesh_small").x0.astype(np.float64), device="cuda")
    handles = [api.Problem(p) for p in probs]
    xs = [g.x.clone() for g in handles]
    torch.cuda.synchronize()
    errors = []

    def work(g, x0, expect):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for _ in range(6):
                    g.x.copy_(x0.reshape(g.x.shape))
                    r = g.solve_lm(3, 9, stream=stream.cuda_stream, persistent=persistent)
                    assert r["E_history"] == expect
        except BaseException as e:                        # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(g, x, w[0])) for g, x, w in zip(handles, xs, want)]
    threads.append(threading.Thread(target=work, args=(f64, x64, want64)))
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for g, w in zip(handles, want):
        np.testing.assert_array_equal(g.x.cpu().numpy(), w[1])
        g.close()
    f64.close()


@pytest.mark.parametrize("kind", ["warp", "poisson", "mesh", "mesh64", "warp64"])
def test_repeated_device_wide_solves_equal_fresh_ones(kind):
    """The counts and slots of the device-wide exchanges go on from launch to launch."""
    from paper_1604_06525_gb300 import api
    f64 = kind.endswith("64")
    cls = api.ProblemF64 if f64 else api.Problem
    prob = make(kind.removesuffix("64"))
    calls = [("gn", 2, 5, {}), ("lm", 3, 4, {}), ("lm", 3, 4, {}), ("gn", 5, 3, {"use_precond": 0}),
             ("gn", 1, 1, {}), ("lm", 2, 6, {"use_graph": 0}), ("gn", 2, 4, {"persistent": -1}), ("lm", 6, 2, {})]
    g = cls(prob)
    x0 = g.x.clone()
    for method, outer, inner, kw in calls:
        fresh = cls(prob)
        want = getattr(fresh, "solve_" + method)(outer, inner, **kw)
        g.x.copy_(x0)
        got = getattr(g, "solve_" + method)(outer, inner, **kw)
        assert got["E_history"] == want["E_history"] and got["pcg_done"] == want["pcg_done"]
        np.testing.assert_array_equal(g.x.cpu().numpy(), fresh.x.cpu().numpy())
        fresh.close()
    lose = g.lib.opt_selftest_lose_block_f64 if f64 else g.lib.opt_selftest_lose_block
    assert lose(g.h) == 0                                 # it was the device-wide loop
    g.close()

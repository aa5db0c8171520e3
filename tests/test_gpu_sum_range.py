"""Dot products of the PCG loop beyond float32's range: scaling a problem by a power of
two scales its solution by it, also where r.z and p.q are sums that no float32 holds
(each thread's share still is one).  The scaled solve may take a float64 quotient for
alpha or beta where the unscaled one takes a float32 pair's; both round to float32, so
they agree to that rounding: TOL as between the routes of a solve."""
import numpy as np
import pytest

from paper_1604_06525_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 2e-6


def scaled(prob, s):
    """Poisson: the images times s.  Mesh: the weights times s (r.z and the energies scale
    by it, the solution stays)."""
    if prob.kind == "poisson":
        return synth.PoissonProblem(prob.W, prob.H, prob.x0 * s, prob.guide * s, prob.mask)
    return synth.MeshProblem(prob.V, prob.urshape, prob.v0, prob.v1, prob.x0, prob.handle_idx, prob.handle_target,
                             float(prob.w_reg * s), float(prob.w_fit * s))


# on chip over one cluster and over the device, single-reduction launches, batch launches
@pytest.mark.parametrize("kind,route", [(k, r) for k in ("poisson_small", "poisson") for r in ("solo", "form1", "batch")] +
                         [("mesh", "solo"), ("mesh", "batch")])
def test_scaled_problem_scales_the_solution(kind, route):
    from paper_1604_06525_gb300 import api
    if kind == "mesh":
        prob = synth.mesh_problem(5, seed=9, handle_frac=0.3)
        prob.handle_target = np.random.default_rng(1).normal(0, 0.5, prob.handle_target.shape).astype(np.float32)
        prob.w_reg, prob.w_fit = 1.0, 4.0
    else:
        # noise: no pixel has more than a small share of a sum
        W, H = (140, 50) if kind == "poisson_small" else (300, 220)
        noise = np.random.default_rng(2).standard_normal((4, H, W)).astype(np.float32)
        prob = synth.PoissonProblem(W, H, np.zeros_like(noise), noise, np.zeros((H, W), np.uint8))

    def solve(p):
        g = api.Problem(p, tile_w=128) if p.kind == "poisson" else api.Problem(p)
        if route == "batch":
            b = api.Batch([g])
            (r,), _ = b.solve_gn(1, 8)
            b.close()
        else:
            r = g.solve_gn(1, 8, pcg_form=int(route == "form1"))
        return g, r

    g, r = solve(prob)
    start = api.Problem(prob)
    rz = start.pcg_init(0.0)
    start.close()
    half = int(np.ceil((131.0 - np.log2(rz)) / 2))               # r.z in [2^131, 2^133): float32 ends at 2^128
    s = 2.0 ** (2 * half if kind == "mesh" else half)
    h, t = solve(scaled(prob, np.float32(s)))
    x, y = g.x.cpu().numpy().astype(np.float64), h.x.cpu().numpy().astype(np.float64)
    if kind != "mesh":
        y /= s
    assert t["pcg_done"] == r["pcg_done"] == 8
    assert np.isfinite(y).all()
    for a, b in zip(x, y):
        assert np.linalg.norm(a - b) <= TOL * max(np.linalg.norm(a), 1e-30)
    for a, b in zip(r["E_history"], t["E_history"]):
        assert abs(a - b / 4.0 ** half) <= 1e-5 * abs(r["E_history"][0])
    g.close()
    h.close()

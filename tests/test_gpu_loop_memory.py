"""What the on-chip PCG loop holds on the device follows the free pixels, not the image,
and a solve for which there is no memory for it takes the launches."""
import numpy as np
import pytest

from paper_1604_06525_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 2e-6          # alpha and beta rounded apart at most (as between the routes of a solve)


def patch(W, H, boxes, kind):
    """Free pixels in some rectangles (x, y, w, h) of a W x H image."""
    mask = np.ones((H, W), np.uint8)
    for x, y, w, h in boxes:
        mask[y:y + h, x:x + w] = 0
    rng = np.random.default_rng(W + H)
    if kind == "warp":
        return synth.warp_problem(W, H, 12, seed=5, max_disp=2.0, mask=mask)
    plane = rng.standard_normal((4, H, W)).astype(np.float32)
    return synth.PoissonProblem(W, H, plane, np.ascontiguousarray(plane[::-1]), mask)


def test_first_solve_of_a_small_patch_takes_little_memory():
    import torch
    from paper_1604_06525_gb300 import api
    prob = patch(2048, 2048, [(500, 700, 300, 200)], "poisson")
    g = api.Problem(prob)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    g.solve_gn(1, 4)
    torch.cuda.synchronize()
    # 60,000 free pixels: 3 records of 16 bytes each, and cells that are partly free
    assert before - torch.cuda.mem_get_info()[0] < 48 << 20
    assert g.lib.opt_selftest_lose_block(g.h) == 0          # the loop ran over the device
    g.close()


# cells with and without neighbours in the list, on all sides, at the image's borders, in
# one cluster and over the device
BOXES = [(64, 64, [(0, 0, 64, 64)]), (200, 90, [(3, 1, 61, 7), (70, 20, 90, 50)]), (33, 9, [(31, 7, 2, 2)]),
         (700, 300, [(31, 7, 34, 10), (100, 0, 500, 300), (650, 290, 50, 10)]), (1030, 40, [(0, 0, 1030, 40)])]


@pytest.mark.parametrize("kind", ["warp", "poisson"])
@pytest.mark.parametrize("W,H,boxes", BOXES)
def test_refused_memory_takes_the_launches(W, H, boxes, kind):
    from paper_1604_06525_gb300 import api
    prob = patch(W, H, boxes, kind)
    for method in ("gn", "lm"):
        on_chip, launches = api.Problem(prob), api.Problem(prob)
        a = getattr(on_chip, "solve_" + method)(2, 7)
        launches.lib.opt_selftest_refuse_allocation()
        b = getattr(launches, "solve_" + method)(2, 7)
        assert b["status"] == "OPT_OK"
        assert launches.lib.opt_selftest_lose_block(launches.h) == 1      # no loop here
        assert a["pcg_done"] == b["pcg_done"] and a["accepted"] == b["accepted"]
        x, y = (p.x.cpu().numpy().astype(np.float64) for p in (on_chip, launches))
        assert np.linalg.norm(x - y) <= TOL * max(np.linalg.norm(y), 1e-30)
        on_chip.close()
        launches.close()

"""Warps whose UrShape is the pixel lattice take wide kernels that do not read it
(GridProb::lattice).  Moving UrShape at one excluded pixel sends the same problem
through the general kernels: no result may change by a bit.
"""
import numpy as np
import pytest

from paper_1604_06525_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("method", ["gn", "lm"])
@pytest.mark.parametrize("W,H", [(128, 8), (129, 9), (300, 57), (1100, 700)])
def test_lattice_warp_equals_general_kernels(W, H, method, form):
    import torch
    from paper_1604_06525_gb300 import api
    mask = synth.random_mask(W, H, 0.2, seed=W)
    mask[H // 2, W // 3] = 1
    got = []
    for moved in (False, True):
        prob = synth.warp_problem(W, H, 12, seed=W + H, max_disp=3.0, mask=mask, x0_noise=0.3)
        prob.urshape += np.float32(5.0)                      # the lattice may lie anywhere
        if moved:
            prob.urshape[0, H // 2, W // 3] += np.float32(0.25)
        members = [api.Problem(prob), api.Problem(prob)]
        batch = api.Batch(members)                           # the launch kernels at every size
        (batch.solve_gn if method == "gn" else batch.solve_lm)(2, 7, pcg_form=form)
        torch.cuda.synchronize()
        got.append(members[0].x.cpu().numpy().copy())
        batch.close()
    assert np.isfinite(got[0]).all()
    np.testing.assert_array_equal(got[0], got[1])


@pytest.mark.parametrize("W,H", [(128, 8), (129, 9), (300, 57), (1100, 700)])
def test_interior_preconditioner_equals_its_planes(W, H):
    """Without a mask the single-reduction kernel forms M^-1 of interior lattice
    pixels itself (with and without a handle); with a mask that excludes nothing it
    reads the planes PCGInit wrote.  The bits agree."""
    import torch
    from paper_1604_06525_gb300 import api
    got = []
    for mask in (None, np.zeros((H, W), np.uint8)):
        prob = synth.warp_problem(W, H, W * H // 60, seed=W + H, max_disp=3.0, mask=mask, x0_noise=0.3)
        members = [api.Problem(prob), api.Problem(prob)]
        batch = api.Batch(members)
        batch.solve_gn(2, 7, pcg_form=1)
        torch.cuda.synchronize()
        got.append(members[0].x.cpu().numpy().copy())
        batch.close()
    np.testing.assert_array_equal(got[0], got[1])

"""The exchanges of the on-chip PCG loops over the device: they complete launch after
launch, a wait that cannot complete gives up within its limit, a solve whose exchange
failed says so without waiting again in its later outer iterations, and the next solve
finds fresh slots whatever its stream."""
import ctypes
import time

import numpy as np
import pytest

from paper_1604_06525_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1604_06525_gb300 import api as api_mod
    api_mod.load_library()
    return api_mod


@pytest.mark.parametrize("kind", [0, 1, 2])
def test_exchange_completes_and_gives_up(api, kind):
    lib = api.load_library()
    t = ctypes.c_int32(-1)
    for rounds in (1, 2, 3, 500):
        assert lib.opt_selftest_resident_exchange(kind, 0, rounds, ctypes.byref(t)) == 0
        assert t.value == 0
    t0 = time.perf_counter()
    assert lib.opt_selftest_resident_exchange(kind, 1, 3, ctypes.byref(t)) == 0
    assert t.value == 1
    assert time.perf_counter() - t0 < 1.0
    assert lib.opt_selftest_resident_exchange(kind, 0, 5, ctypes.byref(t)) == 0
    assert t.value == 0


def test_exchange_selftest_refuses_bad_arguments(api):
    lib = api.load_library()
    t = ctypes.c_int32(-1)
    for kind, absent, rounds in ((-1, 0, 1), (3, 0, 1), (0, 2, 1), (0, 0, 0), (0, 0, 1001)):
        assert lib.opt_selftest_resident_exchange(kind, absent, rounds, ctypes.byref(t)) == 1
    assert lib.opt_selftest_resident_exchange(0, 0, 1, None) == 1
    small = api.Problem(synth.warp_problem(20, 20, 3, seed=1))     # no solve yet: no exchange
    assert lib.opt_selftest_lose_block(small.h) == 1
    small.close()


# more units than one cluster takes, so that the loop runs over the device
@pytest.mark.parametrize("kind,method", [("warp", "lm"), ("poisson", "gn"), ("mesh", "lm"), ("mesh64", "lm"),
                                         ("warp64", "gn")])
def test_failed_exchange_ends_the_solve_and_leaves_the_next_one_alone(api, kind, method):
    import torch
    lib = api.load_library()
    prob = (synth.mesh_problem(5, seed=9, handle_frac=0.05) if kind.startswith("mesh") else
            synth.poisson_problem(300, 200, seed=2) if kind == "poisson" else synth.warp_problem(150, 141, 20, seed=2))
    f64 = kind.endswith("64")
    cls = api.ProblemF64 if f64 else api.Problem
    lose = lib.opt_selftest_lose_block_f64 if f64 else lib.opt_selftest_lose_block
    outer, inner = 6, 5
    fresh = cls(prob)
    want = getattr(fresh, "solve_" + method)(outer, inner)
    g = cls(prob)
    x0 = g.x.clone()
    stream = torch.cuda.Stream()                                   # not ordered with the legacy stream
    for _ in range(3):
        assert getattr(g, "solve_" + method)(outer, inner)["E_history"] == want["E_history"]
        assert lose(g.h) == 0
        g.x.copy_(x0)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        with pytest.raises(api.OptError) as e:
            getattr(g, "solve_" + method)(outer, inner)
        # one wait of 50 ms, not one per outer iteration
        assert time.perf_counter() - t0 < 0.15
        assert e.value.status == 5                                  # OPT_ERR_TIMEOUT
        g.x.copy_(x0)
        torch.cuda.synchronize()
        got = getattr(g, "solve_" + method)(outer, inner, stream=stream.cuda_stream)
        assert got["E_history"] == want["E_history"]
        np.testing.assert_array_equal(g.x.cpu().numpy(), fresh.x.cpu().numpy())
        g.x.copy_(x0)
    g.close()
    fresh.close()

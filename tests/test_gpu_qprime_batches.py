"""The Q' solve at every number of points a block may take (GPU): a point's
arithmetic does not depend on its block, so tiled moments give the first tile's
results bit for bit whatever their count selects, remainders included."""
import numpy as np
import pytest

from paper_2312_06567_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libbgk, cuda_device):
    from paper_2312_06567_gb300 import bgk
    return bgk


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("delta", [0.0, 2.0])
def test_tiled_moments_give_tiled_results(lib, prec, delta):
    """On 152 multiprocessors 8 points per block serve up to 2432 points, 16 up to
    4864, 24 up to 7296, 32 beyond; one point above and below each, and odd counts."""
    wl = W.reduced(W.taylor_green_box(), mesh_n=(3, 1, 1), vel_n=(10, 9, 8)).replace(p=2, delta=delta)
    with lib.Solver(wl, lib.BGK_FP64 if prec == "fp64" else lib.BGK_MIXED) as s:
        s.set_state(W.random_anisotropic_state(wl, seed=8).astype(np.float64 if prec == "fp64" else np.float32))
        m = s.moments()
        q0, it0, st = s.qprime(m)
        assert st == lib.BGK_OK and it0.max() >= 1
        for P in (1, 7, 2431, 2433, 4863, 4865, 7295, 7297, 9727, 9729, 12001):
            reps = -(-P // len(m))
            q, it, st = s.qprime(np.tile(m, (reps, 1))[:P])
            assert st == lib.BGK_OK
            assert np.array_equal(q, np.tile(q0, (reps, 1))[:P]), P
            assert np.array_equal(it, np.tile(it0, reps)[:P]), P

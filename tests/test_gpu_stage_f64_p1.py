"""The FP64 stage at p = 1 on boxes in both of its register forms (GPU): grids of
velocity blocks below and above a wave of one block per multiprocessor, against
the FP64 oracle, over faces and components."""
import numpy as np
import pytest

from oracle import stage as ostage
from paper_2312_06567_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libbgk, cuda_device):
    from paper_2312_06567_gb300 import bgk
    return bgk


@pytest.mark.parametrize("faces", ["periodic", "dirichlet", "specular"])
@pytest.mark.parametrize("delta", [0.0, 2.0])
@pytest.mark.parametrize("mesh_n", [(3, 2, 1), (11, 3, 3), (13, 4, 2)])
def test_rhs_matches_oracle(lib, mesh_n, delta, faces):
    """1, 4 and 4 blocks of elements times 56 velocity blocks on 152 multiprocessors:
    the form of one block per multiprocessor, then that of two.  1e-12 per velocity
    of the largest residual, the parity tests' bound."""
    wl = W.reduced(W.taylor_green_box(), mesh_n=mesh_n, vel_n=(6, 8, 7)).replace(p=1, delta=delta)
    if faces == "dirichlet":
        wl = wl.replace(periodic=(False, True, False), dirichlet={(d, s): (1.0 + 0.1 * d, (0.1 * s, 0.0, -0.1), 1.1)
                                                                  for d in (0, 2) for s in (-1, 1)})
    elif faces == "specular":
        wl = wl.replace(periodic=(False,) * 3, specular=tuple((d, s) for d in range(3) for s in (-1, 1)))
    f = W.random_anisotropic_state(wl, seed=41)
    r_ora, _ = ostage.problem_from_workload(wl).rhs(f)
    with lib.Solver(wl) as s:
        s.set_velocity_blocks(s.velocity_blocks()[2])
        r = s.rhs(f)
    n = wl.n_comp * wl.n_vel
    err = np.max(np.abs(r - r_ora).reshape(n, -1).max(1) / np.abs(r_ora).reshape(n, -1).max(1))
    assert err <= 1e-12, err

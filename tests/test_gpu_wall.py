"""Diffuse-wall densities over orders, face directions and velocity grids: the
FP64 residual of warped meshes with walls across one axis against the oracle.
The grids cover first velocity axes that do and do not divide a block of
threads (up to one below the limit of 128), fewer rows than the blocks take at
once, and rows left over; p > 1 loads element by element, and caller buffers
off the 16-byte boundary make the mixed form's p = 1 do so as well."""
import numpy as np
import pytest

from oracle import curved as ocurved
from paper_2312_06567_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libbgk, cuda_device):
    from paper_2312_06567_gb300 import bgk
    return bgk


def _wl(p, axis, vel_n, delta=0.0):
    wl = W.wavy_periodic_box(p=p, n=(2, 3, 1), vel_n=vel_n, amp=0.06, Pr=1.0).replace(delta=delta)
    return wl.replace(periodic=tuple(d != axis for d in range(3)),
                      diffuse={(axis, -1): ((0.1, 0.2, 0.0), 0.8), (axis, 1): ((0.0, 0.0, -0.1), 1.3)})


def _scale(lib, wl, f, info):
    S, J, fv = lib.curved_metrics(wl, W.node_positions(wl))
    rate = np.max(np.abs(S).sum(axis=(1, 2)) / J) * np.abs(W.velocity_nodes(wl)).max() * (wl.p + 1) ** 2
    return np.abs(f).max() * (rate + 1.0 / info["tau"].min())


@pytest.mark.parametrize("p,axis,vel_n", [(1, 0, (5, 7, 6)), (1, 1, (33, 7, 6)), (1, 2, (127, 6, 7)), (2, 2, (24, 6, 7)),
                                          (2, 0, (8, 13, 9)), (3, 1, (9, 8, 7)), (4, 0, (6, 7, 9)), (4, 2, (7, 6, 6))])
def test_wall_residual_matches_oracle(lib, p, axis, vel_n):
    """Rounding: a wall density sums at most 5334 positive FP64 terms (relative
    error below 5334 * 1.1e-16 = 5.9e-13, traces included), the rest of the
    residual is a few dozen operations of size `scale`."""
    wl = _wl(p, axis, vel_n)
    f = W.random_anisotropic_state(wl, seed=61)
    r_ora, info = ocurved.problem_from_workload(wl, W.node_positions(wl)).rhs(f)
    with lib.Solver(wl, lib.BGK_FP64) as s:
        r = s.rhs(f)
    assert np.max(np.abs(r - r_ora)) <= 1.5e-12 * _scale(lib, wl, f, info)


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_unaligned_mixed_values_give_the_same_walls(lib, axis):
    """The 16-byte loads against single ones: the same values, so the same
    densities up to FP64 rounding; FP32 rounding of the residual remains."""
    import torch
    wl = _wl(1, axis, (10, 7, 6), delta=2.0)
    f = torch.from_numpy(W.random_anisotropic_state(wl, seed=62).astype(np.float32)).cuda()
    buf = torch.empty(f.numel() + 1, dtype=torch.float32, device="cuda")
    off = buf[1:].view(f.shape)
    off.copy_(f)
    _, info = ocurved.problem_from_workload(wl, W.node_positions(wl)).rhs(f.cpu().numpy().astype(np.float64))
    with lib.Solver(wl, lib.BGK_MIXED) as s:
        a, b = torch.empty_like(f), torch.empty_like(f)
        s.stage(f, f, a, 0.0, 0.0, 1.0)                    # out = the residual
        s.stage(f, off, b, 0.0, 0.0, 1.0)
    assert float((a - b).abs().max()) <= 1e-6 * _scale(lib, wl, f.cpu().numpy(), info)

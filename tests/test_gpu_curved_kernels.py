"""The mixed curvilinear stage kernels over orders, components and buffer
alignments (GPU): the residual against the FP64 oracle on warped meshes whose
thread counts are not whole blocks, with both inflow sides and both kinds of
weak face; and caller buffers off the 16-byte boundary, which run without
vector loads, against aligned ones."""
import numpy as np
import pytest

from oracle import curved as ocurved
from paper_2312_06567_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libbgk, cuda_device):
    from paper_2312_06567_gb300 import bgk
    return bgk


def _wl(p, delta, walls):
    wl = W.wavy_periodic_box(p=p, n=(3, 1, 2) if p > 2 else (3, 5, 1), vel_n=(9, 8, 7), amp=0.06, Pr=0.72).replace(delta=delta)
    if walls:                                              # a wall and a farfield across the first axis
        wl = wl.replace(periodic=(False, True, True), diffuse={(0, -1): ((0.0, 0.2, 0.0), 0.8)},
                        dirichlet={(0, 1): (1.1, (0.1, 0.0, -0.1), 1.2)})
    return wl


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("delta", [0.0, 2.0])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_curved_rhs_matches_oracle(lib, p, delta, walls):
    """Per velocity, relative to max|f| (its own or, through the wall and the
    faces, the largest of the block) times the advection rate plus the source:
    FP32 rounding of a few dozen operations, far below 2e-5."""
    wl = _wl(p, delta, walls)
    x = W.node_positions(wl)
    f = W.random_anisotropic_state(wl, seed=21).astype(np.float32)
    pb = ocurved.problem_from_workload(wl, x)
    r_ora, info = pb.rhs(f.astype(np.float64))
    with lib.Solver(wl, lib.BGK_MIXED) as s:
        s.set_qprime_engine(False)                         # the oracle's q' (the FP32 engine stops at 1e-6)
        r = s.rhs(f).astype(np.float64)
    S, J, fv = lib.curved_metrics(wl, x)
    rate = 2.0 * np.max(np.abs(S).sum(axis=(1, 2)) / J) * np.abs(W.velocity_nodes(wl)).max() * (p + 1) ** 2
    scale = np.abs(f).max() * (rate + 1.0 / info["tau"].min())
    assert np.max(np.abs(r - r_ora)) <= 2e-5 * scale / (p + 1)
    fmax = np.abs(f).reshape(wl.n_comp, wl.n_vel, -1).max(axis=2)
    d = np.abs(r - r_ora).reshape(wl.n_comp, wl.n_vel, -1).max(axis=2)
    if not walls:                                          # the wall brings its own values into every velocity
        assert np.max(d / fmax) <= 2e-5 * (rate + 10.0 / info["tau"].min())


@pytest.mark.parametrize("p", [1, 3])
@pytest.mark.parametrize("delta", [0.0, 2.0])
def test_unaligned_caller_buffers(lib, p, delta):
    """The same operations per node with scalar loads: a few ulp of the update
    (compiler contraction) at most."""
    import torch
    wl = _wl(p, delta, True)
    f = torch.from_numpy(W.random_anisotropic_state(wl, seed=22).astype(np.float32)).cuda()
    g = torch.from_numpy(W.random_anisotropic_state(wl, seed=23).astype(np.float32)).cuda()
    n = f.numel()

    def off(t):
        b = torch.empty(n + 1, dtype=torch.float32, device="cuda")
        b[1:].copy_(t.reshape(-1))
        return b[1:].view(t.shape)
    with lib.Solver(wl, lib.BGK_MIXED) as s:
        a, b = torch.empty_like(f), off(f)
        s.stage(g, f, a, 0.75, 0.25, 0.25 * wl.dt())
        s.stage(off(g), off(f), b, 0.75, 0.25, 0.25 * wl.dt())
    assert float((a - b).abs().max()) <= 8 * 2.0 ** -24 * float(f.abs().max())
    assert not torch.equal(a, f)


def _larger_wl(p, delta, walls):
    n = {1: (13, 5, 1), 2: (3, 13, 1), 3: (3, 3, 1), 4: (3, 4, 1)}[p]
    wl = W.wavy_periodic_box(p=p, n=n, vel_n=(9, 8, 7), amp=0.06, Pr=0.72).replace(delta=delta)
    if walls:
        wl = wl.replace(periodic=(False, True, True), diffuse={(0, -1): ((0.0, 0.2, 0.0), 0.8)},
                        dirichlet={(0, 1): (1.1, (0.1, 0.0, -0.1), 1.2)})
    return wl


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("delta", [0.0, 2.0])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_meshes_above_the_node_per_thread_range(lib, p, delta, walls, monkeypatch):
    """The tests above on meshes that the line-group kernel runs whatever their
    faces and components (p = 4 with F and G excepted)."""
    monkeypatch.setitem(globals(), "_wl", _larger_wl)
    test_curved_rhs_matches_oracle(lib, p, delta, walls)
    if walls and p in (1, 3):
        test_unaligned_caller_buffers(lib, p, delta)


def test_no_line_group_geometry_where_no_kernel_reads_it(lib):
    """p = 4 with F and G runs on the node-per-thread kernel: its context holds the
    second component's state beyond a one-component context, not 31 KB per element."""
    import torch
    used = {}
    for delta in (0.0, 2.0):
        wl = W.wavy_periodic_box(p=4, n=(10, 10, 10), vel_n=(2, 2, 2), amp=0.03, Pr=0.72).replace(delta=delta)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        s = lib.Solver(wl, lib.BGK_MIXED)
        used[delta] = free - torch.cuda.mem_get_info()[0]
        s.destroy()
    state = 3 * 1000 * 125 * 8 * 4
    assert used[2.0] <= used[0.0] + state - 1000 * 31000 + (8 << 20)

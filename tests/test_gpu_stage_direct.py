"""The default FP32 stage kernel of box meshes (the line kernel on the copy ring
or reading directly) against the plain one, bit for bit (GPU): every order, one
and two components, every kind of box face, rows that fill a run, leave it short
or have an odd length, and caller buffers off the 16-byte boundary."""
import numpy as np
import pytest

from paper_2312_06567_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libbgk, cuda_device):
    from paper_2312_06567_gb300 import bgk
    return bgk


def _wl(p, mesh_n, delta, faces):
    wl = W.reduced(W.taylor_green_box(), mesh_n=mesh_n, vel_n=(9, 8, 7)).replace(p=p, delta=delta)
    if faces == "dirichlet":
        wl = wl.replace(periodic=(False, True, False), dirichlet={(d, s): (1.0 + 0.1 * d, (0.1 * s, 0.0, -0.1), 1.1)
                                                                  for d in (0, 2) for s in (-1, 1)})
    elif faces == "specular":
        wl = wl.replace(periodic=(False,) * 3, specular=tuple((d, s) for d in range(3) for s in (-1, 1)))
    elif faces == "mixed":
        wl = wl.replace(periodic=(False, True, False), specular=((0, -1), (2, 1)),
                        dirichlet={(0, 1): (1.0, (0.1, 0.0, 0.0), 0.9), (2, -1): (1.1, (0.0, 0.1, 0.0), 1.2)})
    return wl


@pytest.mark.parametrize("faces", ["periodic", "dirichlet", "specular", "mixed"])
@pytest.mark.parametrize("delta", [0.0, 2.0])
@pytest.mark.parametrize("p,n1", [(1, 1), (1, 17), (2, 3), (2, 4), (2, 13), (2, 16), (3, 1), (3, 2), (3, 7), (4, 3)])
def test_default_kernel_equals_plain(lib, p, n1, delta, faces):
    wl = _wl(p, (n1, 2, 3) if n1 < 10 else (n1, 2, 1), delta, faces)
    f = W.random_anisotropic_state(wl, seed=31).astype(np.float32)
    out = []
    for kernel in ("plain", "auto"):
        with lib.Solver(wl, lib.BGK_MIXED) as s:
            s.set_stage_kernel(kernel)
            s.set_state(f)
            r = s.rhs(f)
            s.set_state(f)
            assert s.step(wl.dt(), 2) == lib.BGK_OK
            out.append((r, s.get_state(), s.moments()))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("p,n1", [(1, 5), (3, 4)])
def test_unaligned_caller_buffers_equal_aligned(lib, p, n1):
    import torch
    wl = _wl(p, (n1, 2, 2), 2.0, "periodic")
    f, g = (torch.from_numpy(W.random_anisotropic_state(wl, seed=s).astype(np.float32)).cuda() for s in (32, 33))

    def off(t):
        b = torch.empty(t.numel() + 1, dtype=torch.float32, device="cuda")
        b[1:].copy_(t.reshape(-1))
        return b[1:].view(t.shape)
    with lib.Solver(wl, lib.BGK_MIXED) as s:
        a, b = torch.empty_like(f), off(f)
        s.stage(g, f, a, 0.75, 0.25, 0.25 * wl.dt())
        s.stage(off(g), off(f), b, 0.75, 0.25, 0.25 * wl.dt())
    assert torch.equal(a, b)


def test_tuner_tries_the_direct_form_where_it_is_the_default(lib):
    wl = _wl(2, (7, 2, 2), 0.0, "specular")
    f = W.random_anisotropic_state(wl, seed=34).astype(np.float32)
    with lib.Solver(wl, lib.BGK_MIXED) as s:
        s.set_state(f)
        v, d, ms = s.tune_stage(wl.dt(), reps=1)
        assert v in ("auto", "plain") and ms > 0.0
        assert np.array_equal(s.get_state(), f)


# meshes whose node-per-thread grid is above the waves up to which that kernel is
# the default (below them the test above compares it with itself)
LARGER = [(1, (5, 4, 3)), (1, (17, 3, 3)), (2, (3, 5, 5)), (2, (13, 5, 1)), (2, (16, 4, 1)), (3, (2, 4, 4)), (3, (7, 4, 1)),
          (3, (9, 3, 1)), (4, (3, 4, 2)), (4, (5, 5, 1))]


@pytest.mark.parametrize("faces", ["periodic", "dirichlet", "specular", "mixed"])
@pytest.mark.parametrize("delta", [0.0, 2.0])
@pytest.mark.parametrize("p,mesh_n", LARGER)
def test_line_kernel_by_default_equals_plain(lib, p, mesh_n, delta, faces):
    wl = _wl(p, mesh_n, delta, faces)
    f = W.random_anisotropic_state(wl, seed=35).astype(np.float32)
    out = []
    for kernel in ("plain", "auto"):
        with lib.Solver(wl, lib.BGK_MIXED) as s:
            s.set_velocity_blocks(s.velocity_blocks()[2])
            s.set_stage_kernel(kernel)
            s.set_state(f)
            r = s.rhs(f)
            assert s.step(wl.dt(), 2) == lib.BGK_OK
            out.append((r, s.get_state(), s.moments()))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("faces", ["periodic", "dirichlet", "specular"])
def test_state_beyond_the_cache_at_p1_equals_plain(lib, faces):
    """One wave of the asynchronous kernel's blocks on a state of 49 MB, which that
    kernel runs by default (specular faces excepted)."""
    wl = _wl(1, (32, 1, 1), 2.0, faces).replace(vel_n=(33, 28, 26))
    x = W.node_positions(wl).reshape(-1, 3)
    q = np.stack([1 + 0.1 * np.sin(x[:, 0]), 0.1 * np.cos(x[:, 1]), 0.1 * np.sin(x[:, 2]), 0 * x[:, 0], 1 + 0.05 * np.cos(x[:, 0])], 1)
    out = []
    for kernel in ("plain", "auto"):
        with lib.Solver(wl, lib.BGK_MIXED) as s:
            s.set_stage_kernel(kernel)
            s.set_maxwellian(q)
            assert s.step(wl.dt(), 2) == lib.BGK_OK
            out.append((s.get_state(), s.moments()))
    assert out[0][0].nbytes > 30e6
    for a, b in zip(*out):
        assert np.array_equal(a, b)

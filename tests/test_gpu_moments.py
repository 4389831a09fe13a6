"""Moments, totals and entropy of a stored state against long-double sums
(GPU): point counts that are odd or below one block, first-axis lines shorter
and longer than the kernels' load batches, one and two components, and values
outside the normal range."""
import numpy as np
import pytest

from oracle import stage as ostage
from paper_2312_06567_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libbgk, cuda_device):
    from paper_2312_06567_gb300 import bgk
    return bgk


def _wl(p, mesh_n, vel_n, delta):
    return W.reduced(W.taylor_green_box(), mesh_n=mesh_n, vel_n=vel_n).replace(p=p, delta=delta)


def _reference(wl, f):
    """m[P, 11] in long double, and the sums of magnitudes that scale its errors."""
    u = W.velocity_nodes(wl).astype(np.longdouble)
    w = np.ones(1, dtype=np.longdouble)
    for d in range(3):                                    # k1 fastest
        c = np.full(wl.vel_n[d], (np.longdouble(wl.vel_hi[d]) - wl.vel_lo[d]) / (wl.vel_n[d] - 1))
        c[0] *= 0.5
        c[-1] *= 0.5
        w = (c[:, None] * w[None, :]).reshape(-1)
    psi = [np.ones_like(w), u[:, 0], u[:, 1], u[:, 2], u[:, 0] ** 2, u[:, 1] ** 2, u[:, 2] ** 2, u[:, 0] * u[:, 1],
           u[:, 0] * u[:, 2], u[:, 1] * u[:, 2]]
    F = f[0].reshape(wl.n_vel, -1).astype(np.longdouble)
    m = [(w * s) @ F for s in psi]
    a = [(w * np.abs(s)) @ F for s in psi]
    G = f[1].reshape(wl.n_vel, -1).astype(np.longdouble) if wl.n_comp == 2 else 0 * F
    return np.stack(m + [w @ G], axis=1), np.stack(a + [w @ G], axis=1), w


CASES = [(1, (1, 1, 1), (2, 2, 2), 0.0), (2, (3, 1, 1), (7, 5, 4), 0.0), (2, (5, 1, 1), (9, 3, 8), 2.0),
         (3, (3, 3, 1), (24, 6, 5), 0.0), (4, (5, 1, 1), (17, 4, 3), 2.0), (1, (13, 5, 1), (40, 3, 3), 2.0)]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("case", CASES, ids=[str(i) for i in range(len(CASES))])
def test_moments_totals_entropy_match_long_double_sums(lib, case, prec):
    """Bounds: FP64 sums of n terms lose at most n 2^-53 of the sum of
    magnitudes (n at most the velocities of a block's line sums plus lines);
    16 ulp covers these sizes with the weights' own roundings."""
    wl = _wl(*case)
    f = W.random_anisotropic_state(wl, seed=3)
    if prec == "mixed":
        f = f.astype(np.float32)
    with lib.Solver(wl, lib.BGK_FP64 if prec == "fp64" else lib.BGK_MIXED) as s:
        s.set_state(f)
        m, t, H = s.moments(), s.totals(), s.entropy()
    ref, mag, w = _reference(wl, f)
    n = wl.n_vel
    assert np.all(np.abs(m - ref) <= (16 + 2 * n ** 0.5) * 2.0 ** -53 * np.maximum(mag, 1e-300))
    pb = ostage.problem_from_workload(wl)
    q = wl.p + 1
    Wq = np.einsum("i,j,k->ijk", pb.fr.wq, pb.fr.wq, pb.fr.wq).reshape(-1)
    jac = np.prod([(wl.mesh_hi[d] - wl.mesh_lo[d]) / wl.mesh_n[d] / 2 for d in range(3)])
    Wp = np.tile(Wq, wl.n_elem) * jac
    E = 0.5 * (ref[:, 4] + ref[:, 5] + ref[:, 6]) + ref[:, 10]
    want = np.array([Wp @ ref[:, 0], Wp @ ref[:, 1], Wp @ ref[:, 2], Wp @ ref[:, 3], Wp @ E], dtype=np.float64)
    assert np.all(np.abs(t - want) <= 1e-13 * want[4])
    F = f[0].reshape(n, -1).astype(np.longdouble)
    h = w @ (F * np.log(F))
    assert abs(H - float(Wp @ h)) <= 1e-13 * float(Wp @ (w @ np.abs(F * np.log(F))))
    assert q ** 3 == wl.n_sol


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_values_outside_the_normal_range(lib, prec):
    """Subnormal values count in the entropy, an infinite one makes it and its
    point's moments infinite, a NaN or a zero makes the entropy NaN, and the
    other points' moments stay what they are."""
    wl = _wl(2, (3, 1, 1), (9, 4, 4), 0.0)
    f = W.random_anisotropic_state(wl, seed=4)
    dt = np.float64 if prec == "fp64" else np.float32
    f = f.astype(dt)
    with lib.Solver(wl, lib.BGK_FP64 if prec == "fp64" else lib.BGK_MIXED) as s:
        s.set_state(f)
        m0 = s.moments()
        g = f.copy()
        g[0, 7, 1, 3] = np.finfo(dt).smallest_subnormal * 5
        s.set_state(g)
        F = g[0].reshape(wl.n_vel, -1).astype(np.longdouble)
        _, _, w = _reference(wl, g)
        pb = ostage.problem_from_workload(wl)
        Wq = np.einsum("i,j,k->ijk", pb.fr.wq, pb.fr.wq, pb.fr.wq).reshape(-1)
        jac = np.prod([(wl.mesh_hi[d] - wl.mesh_lo[d]) / wl.mesh_n[d] / 2 for d in range(3)])
        want = float((np.tile(Wq, wl.n_elem) * jac) @ (w @ (F * np.log(F))))
        assert abs(s.entropy() - want) <= 1e-12 * abs(want)
        g[0, 7, 1, 3] = np.inf
        s.set_state(g)
        m = s.moments()
        assert m[1 * wl.n_sol + 3, 0] == np.inf and s.entropy() == np.inf
        keep = np.arange(wl.n_elem * wl.n_sol) != 1 * wl.n_sol + 3
        assert np.array_equal(m[keep], m0[keep])
        g[0, 7, 1, 3] = 0.0
        s.set_state(g)
        assert np.isnan(s.entropy()) and np.all(np.isfinite(s.totals()))
        g[0, 7, 1, 3] = np.nan
        s.set_state(g)
        assert np.isnan(s.entropy())

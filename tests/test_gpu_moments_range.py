"""Moments, totals and entropy where the values' range matters (GPU): dilute
FP32 states whose tails are subnormal, infinite values, velocity grids far
from centred on the gas, values of wide range along the lines, and
values around 1, where ln F is small."""
import numpy as np
import pytest

from oracle import stage as ostage
from paper_2312_06567_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libbgk, cuda_device):
    from paper_2312_06567_gb300 import bgk
    return bgk


def _quadrature(wl):
    """Nodes u[Nu, 3], weights w[Nu] and the points' weights W[P], long double."""
    u = W.velocity_nodes(wl).astype(np.longdouble)
    w = np.ones(1, dtype=np.longdouble)
    for d in range(3):                                    # k1 fastest
        c = np.full(wl.vel_n[d], (np.longdouble(wl.vel_hi[d]) - wl.vel_lo[d]) / (wl.vel_n[d] - 1))
        c[0] *= 0.5
        c[-1] *= 0.5
        w = (c[:, None] * w[None, :]).reshape(-1)
    wq = ostage.problem_from_workload(wl).fr.wq
    jac = np.prod([(wl.mesh_hi[d] - wl.mesh_lo[d]) / wl.mesh_n[d] / 2 for d in range(3)])
    return u, w, np.tile(np.einsum("i,j,k->ijk", wq, wq, wq).reshape(-1), wl.n_elem) * jac


def _entropy(wl, f):
    """The entropy of f's first component and the sum of the magnitudes of its terms, long double."""
    _, w, Wp = _quadrature(wl)
    F = f[0].reshape(wl.n_vel, -1).astype(np.longdouble)
    t = F * np.log(F)
    return Wp @ (w @ t), Wp @ (w @ np.abs(t))


@pytest.mark.parametrize("rho", [1.0, 1e-4, 1e-8, 1e-12])
def test_entropy_of_a_dilute_state_with_subnormal_tails(lib, rho):
    """A Maxwellian whose tail ends just above the smallest subnormal: every
    value counts at its own scale.  Bound: the FP64 sums' 1e-13."""
    wl = W.reduced(W.taylor_green_box(), mesh_n=(2, 1, 1), vel_n=(24, 24, 24)).replace(p=1)
    peak = rho / (2 * np.pi) ** 1.5
    reach = np.sqrt(2 * np.log(peak / 3e-45) / 3)         # |u_d| at the grid's corner
    wl = wl.replace(vel_lo=(-reach,) * 3, vel_hi=(reach,) * 3)
    u = W.velocity_nodes(wl)
    theta = 1 + 0.01 * np.arange(wl.n_elem * wl.n_sol) / (wl.n_elem * wl.n_sol)
    F = rho / (2 * np.pi * theta) ** 1.5 * np.exp(-0.5 * (u ** 2).sum(1)[:, None] / theta)
    f = F.astype(np.float32).reshape(1, wl.n_vel, wl.n_elem, wl.n_sol)
    assert f.min() > 0 and np.mean(f < np.finfo(np.float32).tiny) > 0.005
    with lib.Solver(wl, lib.BGK_MIXED) as s:
        s.set_state(f)
        H = s.entropy()
    want, mag = _entropy(wl, f)
    assert abs(H - float(want)) <= 1e-13 * float(mag)


@pytest.mark.parametrize("delta", [0.0, 2.0])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_an_infinite_value_makes_its_points_moments_and_the_energy_infinite(lib, prec, delta):
    """At a velocity with no zero component, on a grid with a plane u_d = 0 in
    each direction: the moments are infinite with the sign of their weight, as a
    direct sum has them; the other points keep theirs."""
    wl = W.reduced(W.taylor_green_box(), mesh_n=(3, 1, 1), vel_n=(9, 5, 7)).replace(p=2, delta=delta)
    dt = np.float64 if prec == "fp64" else np.float32
    f = W.random_anisotropic_state(wl, seed=4).astype(dt)
    k, at = 7 + 9 * (1 + 5 * 2), 1 * wl.n_sol + 3
    u = W.velocity_nodes(wl)[k]
    assert np.all(u != 0)
    with lib.Solver(wl, lib.BGK_FP64 if prec == "fp64" else lib.BGK_MIXED) as s:
        s.set_state(f)
        m0 = s.moments()
        f[0, k, 1, 3] = np.inf
        s.set_state(f)
        m, t = s.moments(), s.totals()
    psi = [1, u[0], u[1], u[2], u[0] ** 2, u[1] ** 2, u[2] ** 2, u[0] * u[1], u[0] * u[2], u[1] * u[2]]
    assert np.array_equal(m[at, :10], np.inf * np.sign(psi))
    assert abs(m[at, 10] - m0[at, 10]) <= 1e-14 * m0[at, 10]
    assert np.array_equal(np.delete(m, at, 0), np.delete(m0, at, 0))
    assert t[0] == np.inf and t[4] == np.inf and np.array_equal(t[1:4], np.inf * np.sign(u))


def _moments(wl, f):
    """m[P, 11] and the sums of magnitudes that scale its errors, long double."""
    u, w, _ = _quadrature(wl)
    psi = [np.ones_like(w), u[:, 0], u[:, 1], u[:, 2], u[:, 0] ** 2, u[:, 1] ** 2, u[:, 2] ** 2, u[:, 0] * u[:, 1],
           u[:, 0] * u[:, 2], u[:, 1] * u[:, 2]]
    F = f[0].reshape(wl.n_vel, -1).astype(np.longdouble)
    G = f[1].reshape(wl.n_vel, -1).astype(np.longdouble) if wl.n_comp == 2 else 0 * F
    return np.stack([(w * s) @ F for s in psi] + [w @ G], axis=1), np.stack([(w * abs(s)) @ F for s in psi] + [w @ G], axis=1)


@pytest.mark.parametrize("delta", [0.0, 2.0])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("lo,hi", [(-2.0, 60.0), (0.0, 40.0), (3.0, 30.0), (-31.0, -1.0)])
def test_moments_on_grids_far_from_centred(lib, lo, hi, prec, delta):
    """Velocity grids whose middle lies many thermal speeds from the gas.  Bound:
    FP64 sums over n terms, (16 + 2 sqrt n) ulp of the sum of magnitudes."""
    wl = W.reduced(W.taylor_green_box(), mesh_n=(2, 1, 1), vel_n=(64, 9, 8)).replace(p=1, delta=delta)
    wl = wl.replace(vel_lo=(lo, -3.0, lo), vel_hi=(hi, 3.0, hi))
    u = W.velocity_nodes(wl)
    c = np.array([min(max(0.0, lo + 1.0), hi - 1.0), 0.0, min(max(0.0, lo + 1.0), hi - 1.0)])
    rng = np.random.default_rng(1)
    P = wl.n_elem * wl.n_sol
    F = np.exp(-0.5 * ((u[:, None, :] - c - 0.1 * rng.standard_normal((P, 3))) ** 2).sum(-1) / 0.4)
    f = np.stack([F, 0.4 * F])[:wl.n_comp].reshape(wl.n_comp, wl.n_vel, wl.n_elem, wl.n_sol)
    f = np.maximum(f, 1e-30).astype(np.float64 if prec == "fp64" else np.float32)
    with lib.Solver(wl, lib.BGK_FP64 if prec == "fp64" else lib.BGK_MIXED) as s:
        s.set_state(f)
        m = s.moments()
    ref, mag = _moments(wl, f)
    assert np.all(np.abs(m - ref) <= (16 + 2 * wl.n_vel ** 0.5) * 2.0 ** -53 * mag)


@pytest.mark.parametrize("delta", [0.0, 2.0])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("vel_n", [(40, 2, 2), (128, 2, 2), (3, 2, 2)])
def test_moments_of_values_of_wide_range(lib, vel_n, prec, delta):
    """Values over seventeen decades in no order along the lines: a line's sum is
    that of a few of them.  Bound: FP64 sums of n terms round like a random walk,
    1.5 sqrt n ulp of the sum of magnitudes at three sigma, and 6 for the weights."""
    wl = W.reduced(W.taylor_green_box(), mesh_n=(5, 5, 4), vel_n=vel_n).replace(p=3, delta=delta)
    rng = np.random.default_rng(7)
    f = np.exp(-rng.uniform(0.0, 40.0, (wl.n_comp, wl.n_vel, wl.n_elem, wl.n_sol)))
    f = f.astype(np.float64 if prec == "fp64" else np.float32)
    with lib.Solver(wl, lib.BGK_FP64 if prec == "fp64" else lib.BGK_MIXED) as s:
        s.set_state(f)
        m = s.moments()
    ref, mag = _moments(wl, f)
    assert np.all(np.abs(m - ref) <= (6 + 1.5 * wl.n_vel ** 0.5) * 2.0 ** -53 * mag)


CONSTANTS = [1e-30, 3e-7, 0.0635, 0.31, 0.52, 0.74, 0.86, 0.9, 0.9999, 1.0, 1.0000002, 1.06, 1.13, 1.19, 1.9, 7.3, 4e5]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("vel_n", [(24, 3, 2), (128, 2, 2), (5, 2, 2)])
def test_entropy_of_one_value_everywhere(lib, vel_n, prec):
    """Every term has the same rounding, so nothing averages out.  Bound: a
    logarithm good to 4 ulp and FP64 sums of n1 terms, (8 + n1) ulp."""
    wl = W.reduced(W.taylor_green_box(), mesh_n=(1, 1, 1), vel_n=vel_n).replace(p=1)
    dt = np.float64 if prec == "fp64" else np.float32
    with lib.Solver(wl, lib.BGK_FP64 if prec == "fp64" else lib.BGK_MIXED) as s:
        for c in CONSTANTS:
            f = np.full((1, wl.n_vel, wl.n_elem, wl.n_sol), c, dtype=dt)
            s.set_state(f)
            want, mag = _entropy(wl, f)
            assert abs(s.entropy() - want) <= (8 + vel_n[0]) * 2.0 ** -53 * mag, c


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("vel_n", [(24, 5, 4), (128, 3, 2), (3, 2, 2)])
def test_entropy_of_values_of_wide_range(lib, vel_n, prec):
    """Seventeen decades in no order, and a second state around 1."""
    wl = W.reduced(W.taylor_green_box(), mesh_n=(3, 1, 1), vel_n=vel_n).replace(p=2)
    rng = np.random.default_rng(9)
    shape = (1, wl.n_vel, wl.n_elem, wl.n_sol)
    with lib.Solver(wl, lib.BGK_FP64 if prec == "fp64" else lib.BGK_MIXED) as s:
        for lo, hi in ((-40.0, 0.0), (-0.3, 0.3)):
            f = np.exp(rng.uniform(lo, hi, shape)).astype(np.float64 if prec == "fp64" else np.float32)
            s.set_state(f)
            want, mag = _entropy(wl, f)
            assert abs(s.entropy() - want) <= (8 + vel_n[0]) * 2.0 ** -53 * mag

"""The learned guess's training and inference kernels at the edges of their
tiles (GPU): batches below, at and above a chunk of 32 samples and beyond one
chunk per block; inference at tile remainders and on values where e^-z leaves
the held range."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2312_06567_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libbgk, cuda_device):
    from paper_2312_06567_gb300 import bgk
    return bgk


def _net(rng, n, scale=1.0):
    x = np.column_stack([rng.uniform(0.8, 1.2, n), rng.normal(0, 0.1, (n, 3)), rng.uniform(0.9, 1.1, n),
                         rng.uniform(2.9, 3.1, (n, 2)), rng.uniform(0.95, 1.05, n), rng.uniform(0.005, 0.01, n)])
    t = rng.normal(0, 1e-4, (n, 5))
    norm = np.concatenate([[1, 0, 0, 0, 1, 3, 3, 1, 0.0075], [0.1] * 8 + [0.0015], np.zeros(5), np.full(5, 1e-4)])
    params = omlp.init_params(3)
    for b in (1, 3, 5):
        params[b] += rng.normal(0, 0.1, params[b].shape)
    params[0] *= scale
    return x, t, norm, params


@pytest.mark.parametrize("n", [1, 31, 32, 33, 4096, 9800])
def test_gradient_sums_at_chunk_edges(lib, n):
    """FP32 sums over n samples against FP64: each gradient within 1e-5 of the
    largest of its layer (the bound of the gradient test, whatever n)."""
    rng = np.random.default_rng(n)
    x, t, norm, params = _net(rng, n)
    wl = W.reduced(W.periodic_sine_box(), mesh_n=(1, 1, 1), vel_n=(4, 4, 4))
    with lib.Solver(wl) as s:
        s.mlp_weights(load=(params, norm))
        loss_g, grads_g = s.mlp_grad(x, t, bf16=False)
        loss_2, grads_2 = s.mlp_grad(x, t, bf16=False)
    p32 = [np.asarray(p, dtype=np.float32).astype(np.float64) for p in params]
    n32 = norm.astype(np.float32).astype(np.float64)
    xn = (x.astype(np.float32) - n32[:9]) / n32[9:18]
    tn = (t.astype(np.float32) - n32[18:23]) / n32[23:28]
    loss_o, grads_o = omlp.loss_and_grads(p32, xn, tn)
    assert abs(loss_g - loss_o) <= 1e-5 * loss_o
    for go, gg, g2 in zip(grads_o, grads_g, grads_2):
        assert np.max(np.abs(gg - go)) <= 1e-5 * np.max(np.abs(go))
        assert np.array_equal(gg, g2)                      # rows added in a fixed order
    assert loss_2 == loss_g


@pytest.mark.parametrize("n,scale", [(1, 1.0), (127, 1.0), (129, 1.0), (100000, 1.0), (500, 60.0)])
def test_inference_at_tile_edges_and_large_arguments(lib, n, scale):
    """Against the FP64 network with the same BF16 roundings, to the few 1e-3 of
    the output scale a hidden activation's neighbouring BF16 value moves it."""
    rng = np.random.default_rng(n)
    x, t, norm, params = _net(rng, n, scale)
    wl = W.reduced(W.periodic_sine_box(), mesh_n=(1, 1, 1), vel_n=(4, 4, 4))
    with lib.Solver(wl) as s:
        s.mlp_weights(load=(params, norm))
        d = s.mlp_infer(x)
    n32 = norm.astype(np.float32).astype(np.float64)
    p32 = [np.asarray(p, dtype=np.float32).astype(np.float64) for p in params]
    xn = ((x.astype(np.float32) - n32[:9].astype(np.float32)) / n32[9:18].astype(np.float32)).astype(np.float64)
    with np.errstate(over="ignore"):
        y = omlp.forward_bf16(p32, xn)
    err = np.abs((d - n32[18:23]) / n32[23:28] - y)
    assert np.all(np.isfinite(d))
    assert np.max(err) <= 5e-3 * max(1.0, np.abs(y).max())


def test_training_repeats_for_a_seed(lib):
    """Several batches and epochs over a list of samples larger than a copy that
    is staged at once: each epoch takes its own order of the samples, so equal
    seeds give equal weights and losses bit for bit, and another seed others."""
    wl = W.reduced(W.taylor_green_box(), mesh_n=(6, 5, 5), vel_n=(8, 8, 8)).replace(p=3)
    with lib.Solver(wl, lib.BGK_MIXED) as s:
        s.set_state(W.random_anisotropic_state(wl, seed=2).astype(np.float32))
        s.mlp_log(True, 3 * s.n_points)
        s.step(wl.dt(), 1)
        s.mlp_log(False)
        runs = []
        for seed in (5, 5, 5, 6):
            loss = s.mlp_train(epochs=9, batch=900, lr=1e-3, seed=seed)
            runs.append((loss, [p.tobytes() for p in s.mlp_weights()[0]]))
    assert np.isfinite(runs[0][0])
    assert runs[1] == runs[0] and runs[2] == runs[0]
    assert runs[3][1] != runs[0][1]


@pytest.mark.parametrize("z", [-50.0, -300.0, -1e4, -1e10, -1e30])
def test_inference_where_silu_underflows(lib, z):
    """First-layer arguments far below zero, where SiLU is below 1e-19 and a second
    layer of weights 1e12 would show anything larger."""
    params = [np.zeros(p.shape) for p in omlp.init_params(0)]
    params[0][0, :] = 1.0
    params[2][:] = 1e12
    params[3][:] = 1.0
    params[4][:] = 1.0
    norm = np.concatenate([np.zeros(9), np.ones(9), np.zeros(5), np.ones(5)])
    x = np.zeros((300, 9))
    x[:, 0] = z
    x[::7, 0] = 2.0 ** -60                                 # (beside ordinary arguments)
    wl = W.reduced(W.periodic_sine_box(), mesh_n=(1, 1, 1), vel_n=(4, 4, 4))
    with lib.Solver(wl) as s:
        s.mlp_weights(load=(params, norm))
        d = s.mlp_infer(x)
    with np.errstate(over="ignore"):
        y = omlp.forward_bf16([p.astype(np.float32).astype(np.float64) for p in params],
                              x.astype(np.float32).astype(np.float64))
    assert np.max(np.abs(d - y)) <= 5e-3 * np.abs(y).max()

"""The surrogate's gradient kernel at the edges of its tiles (8 rows up to 512
rows, 16 up to 4,096, then 32) against FP64 backpropagation, the standardisation
over many CTAs, and training that repeats to the bit."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2312_05647_gb300 import build as lib_build
    lib_build.build()
    torch.cuda.set_device(0)


def _vec(n):
    return np.concatenate([n["mu_x"], n["sd_x"], [n["mu_y"], n["sd_y"]]])


def _data(rows):
    gen = np.random.default_rng(rows)
    psi = gen.normal(size=(rows, 4))
    return psi, np.sin(psi[:, 0]) + psi[:, 1] * psi[:, 2] + 0.1 * gen.normal(size=rows)


@pytest.mark.parametrize("rows", [1, 7, 8, 9, 512, 513, 2049, 4096, 4097])
def test_gradient_matches_fp64_backprop(rows):
    from paper_2312_05647_gb300 import surrogate as S
    psi, y = _data(rows)
    norm = {"mu_x": np.array([0.1, -0.2, 0.0, 0.3]), "sd_x": np.array([1.0, 0.9, 1.1, 1.2]), "mu_y": 0.2, "sd_y": 0.8}
    p = mlp.init_params(11).astype(np.float32)
    p[mlp.NPAR - 1] = 0.05
    net = S.MLP(seed=0)
    net.set_params(p, _vec(norm))
    loss, g = net.loss_grad(psi, y)
    wl, wg = mlp.loss_grad(p.astype(np.float64), (psi - norm["mu_x"]) / norm["sd_x"], (y - norm["mu_y"]) / norm["sd_y"])
    assert abs(loss - wl) <= 1e-5 * wl
    assert np.abs(g - wg).max() <= 1e-4 * np.abs(wg).max()


@pytest.mark.parametrize("rows", [1, 4096, 4097, 50001])
def test_standardisation_over_many_rows(rows):
    from paper_2312_05647_gb300 import surrogate as S
    psi, y = _data(rows)
    y = y * 30.0 - 20000.0
    net = S.MLP(seed=1)
    net.fit_norm(psi, y)
    np.testing.assert_allclose(net.get_params()[1], _vec(mlp.fit_norm(psi, y)), rtol=1e-12, atol=1e-15)


@pytest.mark.parametrize("batch", [5, 1000, 3000])
def test_training_repeats_to_the_bit(batch):
    import torch
    from paper_2312_05647_gb300 import surrogate as S
    psi, y = _data(6000)
    dp, dy = torch.tensor(psi, device="cuda"), torch.tensor(y, device="cuda")
    runs = []
    for _ in range(2):
        net = S.MLP(seed=3)
        losses = net.train(dp * 1.0, dy * 1.0, steps=40, batch=batch, seed=9, device_data=True)  # data just written
        runs.append((losses, net.get_params()[0]))
    assert np.array_equal(runs[0][0], runs[1][0]) and np.array_equal(runs[0][1], runs[1][1])


@pytest.mark.parametrize("rows", [30, 700])
def test_infinite_residual_gives_an_infinite_gradient(rows):
    """The partials are summed as numbers are: one that overflowed makes the sum
    of its sign infinite, not NaN (the output bias: dL/db3 = sum of dL/df)."""
    from paper_2312_05647_gb300 import surrogate as S
    psi, y = _data(rows)
    y[rows // 2] = 1e39  # beyond FP32 when standardised
    net = S.MLP(seed=0)
    net.set_params(mlp.init_params(11).astype(np.float32), _vec({"mu_x": np.zeros(4), "sd_x": np.ones(4), "mu_y": 0.0, "sd_y": 1.0}))
    loss, g = net.loss_grad(psi, y)
    assert loss == np.inf and g[mlp.NPAR - 1] == -np.inf


def test_standardisation_is_captured_on_a_new_network():
    import ctypes
    import torch
    from paper_2312_05647_gb300 import capi
    from paper_2312_05647_gb300 import surrogate as S
    psi, y = _data(5000)
    dp, dy = torch.tensor(psi, device="cuda"), torch.tensor(y, device="cuda")
    net = S.MLP(seed=1)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        capi.check(capi.lib().mjp_mlp_fit_norm(net._h, ctypes.c_void_p(dp.data_ptr()), ctypes.c_void_p(dy.data_ptr()), 5000,
                                               capi.PTR_DEVICE, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    g.replay()
    torch.cuda.synchronize()
    np.testing.assert_allclose(net.get_params()[1], _vec(mlp.fit_norm(psi, y)), rtol=1e-12, atol=1e-15)

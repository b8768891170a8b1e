"""General rate matrices on two state vectors (the automatic choice where nine
cannot be allocated) give the bits of the chain on nine and of the one-launch
chain."""
import ctypes

import numpy as np
import pytest

import oracle
from test_csr_blocks_gpu import _matrix, _run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2312_05647_gb300 import build as lib_build
    lib_build.build()
    torch.cuda.set_device(0)


def _run_two(rp, col, val, prec, rho0, times, **kw):
    import torch
    import paper_2312_05647_gb300 as mjp
    m = mjp.Model.from_csr(len(rp) - 1, rp, col, val, prec)
    f = getattr(mjp.capi.lib(), "_ZN3mjp13model_csr_twoEP9mjp_model")  # mjp::model_csr_two
    f.restype, f.argtypes = None, [ctypes.c_void_p]
    f(m._h)
    out = m.expv(torch.tensor(rho0, dtype=m.torch_dtype, device="cuda"), times, **kw)
    m.check()
    return out.double().cpu().numpy()


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("n,degrees", [(2, [1]), (33, [0, 3]), (257, [0, 1, 8, 9, 16, 17]), (5003, [7, 8])])
def test_same_bits(n, degrees, prec):
    rp, col, val = _matrix(n, degrees, n)
    gen = np.random.default_rng(n + 1)
    rho0 = gen.random(n)
    rho0 /= rho0.sum()
    om = oracle.expv(oracle.CSR(rp, col, val), rho0, [0.0])[1]["omega"]
    times = np.array([0.0, 0.01, 0.97, 4.4, 70.0, 71.0, 300.0]) / om
    for kw in ({}, {"trunc": 1, "tol": 1e-10}):
        two = _run_two(rp, col, val, prec, rho0, times, **kw)
        assert np.array_equal(two, _run(rp, col, val, prec, rho0, times, 0, **kw))
        assert np.array_equal(two, _run(rp, col, val, prec, rho0, times, 2, **kw))


def test_a_ring_that_leaves_the_l2_is_not_taken():
    """3 million states, random FP64 entries, one time: nine vectors took 1.2 times as long as two."""
    import torch
    import paper_2312_05647_gb300 as mjp
    n, d = 3000000, 4
    gen = np.random.default_rng(5)
    off = np.sort(gen.integers(0, n // d - 1, (n, d)) + np.arange(d) * (n // d), axis=1) + 1
    col = np.sort((np.arange(n)[:, None] + off) % n, axis=1).ravel().astype(np.int32)
    rp, val = np.arange(n + 1, dtype=np.int64) * d, gen.lognormal(0.0, 1.0, n * d)
    rho0 = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    f = getattr(mjp.capi.lib(), "_ZN3mjp13model_csr_twoEP9mjp_model")
    f.restype, f.argtypes = None, [ctypes.c_void_p]
    ms, outs = [], []
    for two in (False, True):
        m = mjp.Model.from_csr(n, rp, col, val, 2)
        if two:
            f(m._h)
        om = m.expv(rho0, [1e-9], info=True)[1]["omega"]
        best = np.inf
        for _ in range(4):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            a.record()
            out = m.expv(rho0, [60.0 / om])
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
        outs.append(out)
    assert torch.equal(outs[0], outs[1])
    assert ms[0] <= 1.05 * ms[1], ms

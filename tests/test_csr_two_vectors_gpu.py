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

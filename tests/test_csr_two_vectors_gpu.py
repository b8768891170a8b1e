"""General rate matrices on two state vectors (MJP_OPT_CHAIN = 1, and the
automatic choice where nine cannot be allocated) give the bits of the chain on
nine and of the one-launch chain."""
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
        two = _run(rp, col, val, prec, rho0, times, 1, **kw)
        assert np.array_equal(two, _run(rp, col, val, prec, rho0, times, 0, **kw))
        assert np.array_equal(two, _run(rp, col, val, prec, rho0, times, 2, **kw))

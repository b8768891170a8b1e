"""General rate matrices at the edges of the chain's blocks of eight jumps and
of its preloaded entries: K around multiples of 8, ragged rows from no
transition to several hundred, windows of several times in one block, both
truncation rules, against the oracle and the one-launch chain."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
TOL = {1: 1e-6, 2: 1e-12}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2312_05647_gb300 import build as lib_build
    lib_build.build()
    torch.cuda.set_device(0)


def _matrix(n, degrees, seed):
    gen = np.random.default_rng(seed)
    deg = np.minimum(gen.choice(degrees, n), n - 1)
    rp = np.concatenate([[0], np.cumsum(deg)])
    col = np.concatenate([np.sort((i + 1 + gen.choice(n - 1, d, replace=False)) % n) for i, d in enumerate(deg)] + [np.zeros(0)])
    return rp, col.astype(np.int32), gen.lognormal(0.0, 1.0, rp[-1])


def _run(rp, col, val, prec, rho0, times, chain, **kw):
    import torch
    import paper_2312_05647_gb300 as mjp
    m = mjp.Model.from_csr(len(rp) - 1, rp, col, val, prec)
    m.set_option(mjp.OPT_CHAIN, chain)
    out = m.expv(torch.tensor(rho0, dtype=m.torch_dtype, device="cuda"), times, **kw)
    m.check()
    return out.double().cpu().numpy()


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("n,degrees", [(2, [1]), (33, [0, 3]), (257, [0, 1, 8, 9, 16, 17]), (1000, [1, 400]), (5003, [7, 8])])
def test_blocks_and_ragged_rows(n, degrees, prec):
    rp, col, val = _matrix(n, degrees, n)
    gen = np.random.default_rng(n + 1)
    rho0 = gen.random(n)
    rho0 /= rho0.sum()
    om = oracle.expv(oracle.CSR(rp, col, val), rho0, [0.0])[1]["omega"]
    # x = 0, tiny, and values whose K = floor(x + 6 sqrt x) + 1 is 7, 8, 9, 16, 17, 121 and beyond.
    x = np.array([0.0, 0.01, 0.8, 0.97, 1.2, 4.0, 4.4, 70.0, 71.0, 300.0])
    times = x / om
    for kw in ({}, {"trunc": 1, "tol": 1e-10}):
        a = _run(rp, col, val, prec, rho0, times, 0, **kw)
        assert np.array_equal(a, _run(rp, col, val, prec, rho0, times, 2, **kw))
        ref, _ = oracle.expv(oracle.CSR(rp, col, val), rho0, times, **({"mode": 1, "tol": 1e-10} if kw else {}))
        assert np.abs(a - ref).max() <= TOL[prec]

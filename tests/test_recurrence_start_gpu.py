"""Windows without a stored copy of their weights (an arena of one element) run
Algorithm 2's recurrence from P_L, which is far below FP32's normal range
for x = Omega t around 100: the recurrence still starts from the right value."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2312_05647_gb300 import build as lib_build
    lib_build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("chain", [0, 1])
@pytest.mark.parametrize("kind,dims,th", [(1, [40], [7.0, 0.6]), (2, [30], [9.0, 0.7, 2.0, 1.0]), (3, [21, 20], [3.0, 0.5, 1.5, 0.2])])
def test_fp32_recurrence_around_x_100(kind, dims, th, chain):
    import torch
    import paper_2312_05647_gb300 as mjp
    n = int(np.prod(dims)) * (2 if kind == 2 else 1)
    rho0 = synth.delta(n, 0)
    csr = oracle.build_model(kind, dims, th)
    omega = oracle.expv(csr, rho0, [1e-3])[1]["omega"]
    times = np.array([60.0, 85.0, 95.0, 99.0, 103.0, 106.0, 109.5, 110.5, 112.0, 118.0, 125.0, 150.0, 210.0, 300.0]) / omega
    m = mjp.Model(kind, dims, th, 1)
    m.set_option(mjp.OPT_CHAIN, chain)
    m.set_option(mjp.OPT_ARENA, 1)
    out = m.expv(torch.tensor(rho0, dtype=torch.float32, device="cuda"), times).double().cpu().numpy()
    m.check()
    ref = oracle.expv(csr, rho0, times)[0]
    # The FP32 chain's own tolerance; the weights sum to 1 within a few FP32 roundings.
    assert np.abs(out - ref).max() <= 1e-6
    assert np.abs(out.sum(axis=1) - 1.0).max() <= 1e-6

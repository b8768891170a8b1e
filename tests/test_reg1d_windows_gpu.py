"""expv_series of larger birth-death models (csrc/stencil_reg1d.cu): the kernel
for overlapping windows and the one that keeps the sums of a round's only window
in registers, both with the bits of the shared-memory chain, on either side of
the rule that chooses between them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2312_05647_gb300 import build as lib_build
    lib_build.build()
    torch.cuda.set_device(0)


# x = Omega t of the times: one, apart, touching, overlapping, all together.
TIMES = [[300.0], [3.0, 2000.0], [100.0, 400.0, 900.0], [400.0, 420.0, 700.0], list(np.linspace(300.0, 400.0, 10))]


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("x", TIMES)
@pytest.mark.parametrize("n", [513, 2000, 9000])
def test_same_bits_as_the_shared_memory_chain(n, x, prec):
    import torch
    import paper_2312_05647_gb300 as mjp
    theta = [0.4 * n, 1.0]
    times = np.asarray(x) / (1.1 * (theta[0] + theta[1] * (n - 2)))
    out = []
    for chain in (0, 1):
        m = mjp.Model(1, [n], theta, prec)
        m.set_option(mjp.OPT_CHAIN, chain)
        rho0 = torch.tensor(np.random.default_rng(n).dirichlet(np.ones(n)), dtype=m.torch_dtype, device="cuda")
        out.append(m.expv(rho0, times).cpu().numpy())
        m.check()
    assert np.array_equal(out[0], out[1])


def test_overlapping_windows_are_not_slower():
    """3,955 states FP32, 16 times close together against the last of them alone (independent of the clock)."""
    import torch
    import paper_2312_05647_gb300 as mjp
    n = 3955
    times = np.linspace(0.8 * 449, 449, 16) / (1.1 * (7.0 + 0.6 * (n - 1)))
    rho0 = torch.full((n,), 1.0 / n, dtype=torch.float32, device="cuda")
    m = mjp.Model(1, [n], [7.0, 0.6], 1)
    ms = []
    for t in (times, times[-1:]):
        m.expv(rho0, t)
        best = np.inf
        for _ in range(8):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            a.record()
            m.expv(rho0, t)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
    m.check()
    assert ms[0] <= 8.15 * ms[1], ms  # 7.43 to 7.49; 8.88 to 8.95 where the kernel spills

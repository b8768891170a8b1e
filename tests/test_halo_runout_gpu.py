"""Halo waits of the register/tile chain that run out at the first hand-over of
a long chain (thousands of hand-overs follow, more bytes than an mbarrier
counts): an error status, and the same handle works again afterwards."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
MP, AR = 3, 5


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2312_05647_gb300 import build as lib_build
    lib_build.build()
    torch.cuda.set_device(0)


def _setup(kind, dims, prec):
    import paper_2312_05647_gb300 as mjp
    th = [3.0, 0.5, 1.5, 0.2] if kind == MP else [4.0, 0.5, 0.6, 0.1, 0.4, 0.05]
    n = int(np.prod(dims)) * (2 if kind == AR else 1)
    omega = oracle.expv(oracle.build_model(kind, dims, th), synth.delta(n, 0), [1e-3])[1]["omega"]
    return mjp, mjp.Model(kind, dims, th, prec), n, th, np.array([6000.0, 12000.0]) / omega


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind,dims", [(MP, [120, 90]), (AR, [40, 61])])
def test_long_series_after_a_wait_that_ran_out(kind, dims, prec):
    import torch
    mjp, m, n, _, times = _setup(kind, dims, prec)
    rho0 = torch.tensor(synth.delta(n, 0), dtype=m.torch_dtype, device="cuda")
    want = m.expv(rho0, times)
    m.check()
    m.set_option(mjp.OPT_WAIT_LIMIT, 0)
    m.expv(rho0, times)
    with pytest.raises(mjp.MJPError) as e:
        m.check()
    assert e.value.code == -5
    m.set_option(mjp.OPT_WAIT_LIMIT, 1 << 24)
    assert torch.equal(m.expv(rho0, times), want)
    m.check()


@pytest.mark.parametrize("prec", [1, 2])
def test_long_log_likelihood_after_a_wait_that_ran_out(prec):
    mjp, m, n, th, times = _setup(AR, [40, 120], prec)
    obs = mjp.Obs(n, times, [([np.array([s]) for s in (0, 1, 45)], np.ones(3))] * 2, synth.delta(n, 0))
    ths = np.asarray([th])
    want = mjp.loglik(m, obs, ths)
    m.check()

    m.set_option(mjp.OPT_WAIT_LIMIT, 0)
    with pytest.raises(mjp.MJPError) as e:  # a call that returns host data returns the status
        mjp.loglik(m, obs, ths)
    assert e.value.code == -5
    m.set_option(mjp.OPT_WAIT_LIMIT, 1 << 24)
    assert np.array_equal(mjp.loglik(m, obs, ths), want)
    m.check()

"""The register/tile jump chain (csrc/stencil_tile.cuh: the automatic choice of
expv_series for two-state, mRNA/protein and autoregulatory models and of
loglik for birth-death, autoregulatory and FP64 models) against the
shared-memory chain (MJP_OPT_CHAIN = 1) and the oracle, at the edges of its
runs, tiles, halos and observation slots."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
BD, TS, MP, AR = 1, 2, 3, 5
U32 = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2312_05647_gb300 import build as lib_build
    lib_build.build()
    torch.cuda.set_device(0)


def _size(kind, dims):
    return int(np.prod(dims)) * (2 if kind in (TS, AR) else 1)


def _theta(kind):
    return {BD: [7.0, 0.6], TS: [9.0, 0.7, 2.0, 1.0], MP: [3.0, 0.5, 1.5, 0.2], AR: [4.0, 0.5, 0.6, 0.1, 0.4, 0.05]}[kind]


def _omega(kind, dims, th):
    m = oracle.build_model(kind, dims, th)
    return oracle.expv(m, synth.delta(_size(kind, dims), 0), [1e-3])[1]["omega"]


def _times(kind, dims, x):
    return np.asarray(x) / max(_omega(kind, dims, _theta(kind)), 1e-9)


def _model(kind, dims, prec, chain, **opts):
    import paper_2312_05647_gb300 as mjp
    m = mjp.Model(kind, dims, _theta(kind), prec)
    m.set_option(mjp.OPT_CHAIN, chain)
    for k, v in opts.items():
        m.set_option(getattr(mjp, k), v)
    return m


def _expv(kind, dims, prec, chain, rho0, times, trunc=0, tol=0.0, **opts):
    import torch
    m = _model(kind, dims, prec, chain, **opts)
    out = m.expv(torch.tensor(rho0, dtype=m.torch_dtype, device="cuda"), times, trunc=trunc, tol=tol)
    m.check()
    return out.double().cpu().numpy()


def _close_expv(a, b, prec):
    """FP64: the same operations.  FP32: the same chain; each output is a sum of
    products, rounded per jump on one side (Kahan: 2 u plus u per product) and
    in chains of at most 16 multiply-adds on the other (16 u plus 2 u)."""
    if prec == 2:
        assert np.array_equal(a, b)
    else:
        assert np.all(np.abs(a - b) <= 21 * U32 * np.abs(b) + 1e-36)


SERIES = [(TS, [2]), (TS, [37]), (TS, [300]), (TS, [900]), (MP, [2, 1]), (MP, [21, 1]), (MP, [33, 7]), (MP, [18, 199]),
          (MP, [120, 90]), (MP, [201, 64]), (AR, [2, 2]), (AR, [13, 2]), (AR, [25, 30]), (AR, [40, 61])]


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind,dims", SERIES)
def test_expv_equals_shared_memory_chain(kind, dims, prec):
    n = _size(kind, dims)
    gen = np.random.default_rng(n + prec)
    rho0 = gen.random(n)
    rho0 /= rho0.sum()
    times = _times(kind, dims, [30.0, 0.0, 3.0, 140.0, 31.0, 31.0, 62.0])
    _close_expv(_expv(kind, dims, prec, 0, rho0, times), _expv(kind, dims, prec, 1, rho0, times), prec)


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind,dims,nt", [(TS, [60], 256), (MP, [90, 80], 60), (AR, [30, 40], 90)])
def test_expv_many_overlapping_times(kind, dims, nt, prec):
    """More overlapping windows than shared accumulators, weight chunks of every length."""
    n = _size(kind, dims)
    rho0 = synth.delta(n, 0)
    times = _times(kind, dims, np.linspace(0.0, 400.0, nt))
    _close_expv(_expv(kind, dims, prec, 0, rho0, times), _expv(kind, dims, prec, 1, rho0, times), prec)


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind,dims", [(TS, [45]), (MP, [60, 75]), (AR, [20, 33])])
def test_expv_without_stored_weights_and_tolerance_rule(kind, dims, prec):
    """The in-kernel recurrence (an arena of one element) and K by tolerance."""
    n = _size(kind, dims)
    rho0 = np.full(n, 1.0 / n)
    times = _times(kind, dims, [0.0, 2.0, 47.0, 90.0])
    a = _expv(kind, dims, prec, 0, rho0, times, OPT_ARENA=1)
    _close_expv(a, _expv(kind, dims, prec, 1, rho0, times, OPT_ARENA=1), prec)
    a = _expv(kind, dims, prec, 0, rho0, times, trunc=1, tol=1e-9)
    _close_expv(a, _expv(kind, dims, prec, 1, rho0, times, trunc=1, tol=1e-9), prec)


@pytest.mark.parametrize("prec", [1, 2])
def test_expv_time_above_the_cap_is_reported_and_has_no_result(prec):
    import torch
    import paper_2312_05647_gb300 as mjp
    dims = [30, 40]
    m = _model(MP, dims, prec, 0, OPT_K_CAP=100)
    rho0 = synth.delta(1200, 0)
    times = _times(MP, dims, [20.0, 400.0])
    out = m.expv(torch.tensor(rho0, dtype=m.torch_dtype, device="cuda"), times)
    with pytest.raises(mjp.MJPError) as e:
        m.check()
    assert e.value.code == -6
    out = out.double().cpu().numpy()
    ref = _expv(MP, dims, prec, 1, rho0, times[:1])
    _close_expv(out[:1], ref, prec)
    assert np.isnan(out[1]).all()


def test_expv_hand_over_wait_that_runs_out_is_reported():
    """A cluster whose halo waits give up at once: an error status, and the model works again afterwards."""
    import torch
    import paper_2312_05647_gb300 as mjp
    dims = [120, 90]
    rho0 = synth.delta(10800, 0)
    times = _times(MP, dims, [200.0])
    m = _model(MP, dims, 1, 0, OPT_WAIT_LIMIT=0)
    r = torch.tensor(rho0, dtype=torch.float32, device="cuda")
    m.expv(r, times)
    with pytest.raises(mjp.MJPError) as e:
        m.check()
    assert e.value.code == -5
    m.set_option(mjp.OPT_WAIT_LIMIT, 1 << 24)
    out = m.expv(r, times)
    m.check()
    _close_expv(out.double().cpu().numpy(), _expv(MP, dims, 1, 1, rho0, times), 1)


def _obs(kind, dims, nt, groups, gen):
    """Groups of one or two states, some states twice."""
    n = _size(kind, dims)
    out = []
    for _ in range(nt):
        k = min(n, groups)
        first = gen.choice(n, size=k, replace=False)
        mem = [np.array([s]) if gen.random() < 0.5 else np.array([s, gen.integers(0, n)]) for s in first]
        out.append((mem, gen.integers(1, 5, k).astype(float)))
    return out


# Box, observation groups per time, thetas: one CTA or clusters, 1 .. 8 groups a thread, several CTAs per SM.
LOGLIK = [(BD, [1], 1, 3), (BD, [2], 2, 1), (BD, [33], 20, 700), (BD, [64], 60, 1), (BD, [1001], 200, 2), (BD, [5000], 40, 1),
          (TS, [2], 3, 2), (TS, [37], 25, 1), (TS, [131], 150, 300), (TS, [700], 90, 1), (MP, [21, 1], 9, 2), (MP, [33, 7], 30, 1),
          (MP, [18, 199], 40, 1), (MP, [90, 60], 30, 160), (AR, [2, 2], 3, 1), (AR, [13, 2], 20, 5), (AR, [25, 30], 160, 160),
          (AR, [40, 61], 400, 1), (AR, [40, 120], 330, 3)]


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind,dims,groups,B", LOGLIK)
def test_loglik_equals_shared_memory_chain(kind, dims, groups, B, prec):
    import paper_2312_05647_gb300 as mjp
    n = _size(kind, dims)
    gen = np.random.default_rng(n + 7 * B)
    rho0 = gen.random(n)
    rho0 /= rho0.sum()
    times = _times(kind, dims, [12.0, 0.0, 30.0, 31.0, 60.0, 90.0, 140.0])
    ob = _obs(kind, dims, len(times), groups, gen)
    obs = mjp.Obs(n, times, ob, rho0)
    nobs = sum(float(c.sum()) for _, c in ob)
    th = np.asarray(_theta(kind)) * gen.uniform(0.8, 1.2, size=(B, len(_theta(kind))))
    ll = {}
    for chain in (0, 1):
        m = _model(kind, dims, prec, chain)
        ll[chain] = mjp.loglik(m, obs, th)
        m.check()
    # Equal chains and the same sums per group: a group's probability differs
    # by at most its compensation's rounding (2 u per observation in FP32).
    # (a state without mass gives -inf on both sides).
    fine = np.isfinite(ll[1])
    assert np.array_equal(ll[0][~fine], ll[1][~fine])
    assert np.all(np.abs(ll[0][fine] - ll[1][fine]) <= nobs * (2 * U32 if prec == 1 else 1e-14) + 1e-12)


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind,dims", [(BD, [70]), (TS, [52]), (MP, [26, 31]), (AR, [12, 19])])
def test_loglik_matches_oracle(kind, dims, prec):
    import paper_2312_05647_gb300 as mjp
    n = _size(kind, dims)
    gen = np.random.default_rng(n)
    rho0 = synth.delta(n, 0)
    times = _times(kind, dims, [20.0, 55.0, 300.0])
    th = _theta(kind)
    m = oracle.build_model(kind, dims, th)
    # States that carry mass at their time.
    p = oracle.expv(m, rho0, times)[0]
    ob = []
    for i in range(3):
        top = np.argsort(p[i])[::-1][:12]
        ob.append(([np.array([s]) for s in top], gen.integers(1, 6, len(top)).astype(float)))
    obs = mjp.Obs(n, times, ob, rho0)
    nobs = sum(float(c.sum()) for _, c in ob)
    ll = mjp.loglik(_model(kind, dims, prec, 0), obs, np.asarray([th]))[0]
    ref = oracle.loglik(m, rho0, times, ob)
    assert abs(ll - ref) <= nobs * (5e-6 if prec == 1 else 1e-12)

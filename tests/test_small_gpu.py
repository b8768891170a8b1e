"""The small-model chain (csrc/stencil_small.cu: the automatic choice of
expv_series for birth-death and two-state models of at most 512 states) against
the shared-memory chain (MJP_OPT_CHAIN = 1) at the edges of its warps, blocks
and weight chunks, and its first and smallest sizes against the oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
BD, TS = 1, 2
U32 = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2312_05647_gb300 import build as lib_build
    lib_build.build()
    torch.cuda.set_device(0)


def _theta(kind):
    return [7.0, 0.6] if kind == BD else [9.0, 0.7, 2.0, 1.0]


def _n(kind, dims):
    return dims[0] * (2 if kind == TS else 1)


def _times(kind, dims, x):
    om = oracle.expv(oracle.build_model(kind, dims, _theta(kind)), synth.delta(_n(kind, dims), 0), [1e-3])[1]["omega"]
    return np.asarray(x) / max(om, 1e-9)


def _expv(kind, dims, prec, chain, rho0, times, trunc=0, tol=0.0, check=True, **opts):
    import torch
    import paper_2312_05647_gb300 as mjp
    m = mjp.Model(kind, dims, _theta(kind), prec)
    m.set_option(mjp.OPT_CHAIN, chain)
    for k, v in opts.items():
        m.set_option(getattr(mjp, k), v)
    out = m.expv(torch.tensor(rho0, dtype=m.torch_dtype, device="cuda"), times, trunc=trunc, tol=tol)
    if check:
        m.check()
    return out.double().cpu().numpy(), m


def _same(a, b, prec):
    """FP64: the same operations.  FP32: the same chain, sums of 8 products in a
    fused chain and a Kahan step against a Kahan step per product (11 u + 3 u)."""
    if prec == 2:
        assert np.array_equal(a, b)
    else:
        assert np.all(np.abs(a - b) <= 14 * U32 * np.abs(b) + 1e-36)


SIZES = [(BD, [1]), (BD, [2]), (BD, [31]), (BD, [33]), (BD, [64]), (BD, [512]), (TS, [2]), (TS, [16]), (TS, [37]), (TS, [131]),
         (TS, [256])]


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind,dims", SIZES)
def test_equals_shared_memory_chain(kind, dims, prec):
    n = _n(kind, dims)
    gen = np.random.default_rng(n)
    rho0 = gen.random(n)
    rho0 /= rho0.sum()
    # K from 0 over the edges of blocks (8) and chunks (32), windows that overlap, coincide and leave gaps.
    times = _times(kind, dims, [30.0, 0.0, 0.5, 3.0, 140.0, 31.0, 31.0, 600.0])
    a, _ = _expv(kind, dims, prec, 0, rho0, times)
    b, _ = _expv(kind, dims, prec, 1, rho0, times)
    _same(a, b, prec)


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind,dims,nt", [(BD, [20], 256), (TS, [15], 256), (BD, [100], 60)])
def test_many_times_weights_by_recurrence_and_tolerance(kind, dims, nt, prec):
    n = _n(kind, dims)
    rho0 = synth.delta(n, 0)
    times = _times(kind, dims, np.linspace(0.0, 400.0, nt))
    for kw in ({}, {"OPT_ARENA": 1}, {"trunc": 1, "tol": 1e-9}):
        a, _ = _expv(kind, dims, prec, 0, rho0, times, **kw)
        b, _ = _expv(kind, dims, prec, 1, rho0, times, **kw)
        _same(a, b, prec)


@pytest.mark.parametrize("prec", [1, 2])
def test_time_above_the_cap_has_no_result(prec):
    import paper_2312_05647_gb300 as mjp
    rho0 = synth.delta(40, 0)
    times = _times(BD, [40], [20.0, 400.0])
    out, m = _expv(BD, [40], prec, 0, rho0, times, check=False, OPT_K_CAP=100)
    with pytest.raises(mjp.MJPError) as e:
        m.check()
    assert e.value.code == -6
    _same(out[:1], _expv(BD, [40], prec, 1, rho0, times[:1])[0], prec)
    assert np.isnan(out[1]).all()


@pytest.mark.parametrize("prec,tol", [(1, 1e-6), (2, 1e-12)])
@pytest.mark.parametrize("kind,dims", [(BD, [2]), (BD, [64]), (BD, [300]), (TS, [9]), (TS, [131])])
def test_matches_oracle(kind, dims, prec, tol):
    n = _n(kind, dims)
    rho0 = synth.delta(n, 0)
    times = _times(kind, dims, [0.3, 7.0, 1500.0])
    out, _ = _expv(kind, dims, prec, 0, rho0, times)
    ref = oracle.expv(oracle.build_model(kind, dims, _theta(kind)), rho0, times)[0]
    assert np.abs(out - ref).max() <= tol

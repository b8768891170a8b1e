"""FP32 transient distributions: every product P_k rho_k has a Kahan step of its
own in every chain, so the register/tile chain and the small-model chain give
the bits of the shared-memory chain (MJP_OPT_CHAIN = 1)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
BD, TS, MP, AR = 1, 2, 3, 5


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2312_05647_gb300 import build as lib_build
    lib_build.build()
    torch.cuda.set_device(0)


def _theta(kind):
    return {BD: [7.0, 0.6], TS: [9.0, 0.7, 2.0, 1.0], MP: [3.0, 0.5, 1.5, 0.2], AR: [4.0, 0.5, 0.6, 0.1, 0.4, 0.05]}[kind]


def _expv(kind, dims, chain, rho0, x, **opts):
    import torch
    import paper_2312_05647_gb300 as mjp
    om = oracle.expv(oracle.build_model(kind, dims, _theta(kind)), rho0, [1e-3])[1]["omega"]
    m = mjp.Model(kind, dims, _theta(kind), 1)
    m.set_option(mjp.OPT_CHAIN, chain)
    for k, v in opts.items():
        m.set_option(getattr(mjp, k), v)
    out = m.expv(torch.tensor(rho0, dtype=torch.float32, device="cuda"), np.asarray(x) / max(om, 1e-9))
    m.check()
    return out.cpu().numpy()


# Small-model chain (up to 512 states), then one CTA and clusters of the register/tile chain.
BOXES = [(BD, [1]), (BD, [33]), (BD, [512]), (TS, [16]), (TS, [256]), (TS, [300]), (TS, [900]), (MP, [33, 7]), (MP, [18, 199]),
         (MP, [120, 90]), (MP, [201, 64]), (AR, [13, 2]), (AR, [25, 30]), (AR, [40, 61])]


@pytest.mark.parametrize("kind,dims", BOXES)
def test_same_bits_as_the_shared_memory_chain(kind, dims):
    n = int(np.prod(dims)) * (2 if kind in (TS, AR) else 1)
    gen = np.random.default_rng(n)
    rho0 = gen.random(n)
    rho0 /= rho0.sum()
    # Windows that begin and end at every place of a block, coincide, overlap and leave gaps.
    x = [30.0, 0.0, 0.5, 3.0, 140.0, 31.0, 31.0, 600.0, *np.linspace(150.0, 190.0, 9)]
    for opts in ({}, {"OPT_ARENA": 1}):
        assert np.array_equal(_expv(kind, dims, 0, rho0, x, **opts), _expv(kind, dims, 1, rho0, x, **opts))


@pytest.mark.parametrize("kind,dims,nt", [(BD, [90], 200), (TS, [60], 256), (MP, [90, 80], 60), (AR, [30, 40], 90)])
def test_same_bits_with_more_windows_than_shared_accumulators(kind, dims, nt):
    n = int(np.prod(dims)) * (2 if kind in (TS, AR) else 1)
    rho0, x = synth.delta(n, 0), np.linspace(0.0, 400.0, nt)
    assert np.array_equal(_expv(kind, dims, 0, rho0, x), _expv(kind, dims, 1, rho0, x))

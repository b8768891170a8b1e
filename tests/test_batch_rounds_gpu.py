"""Register-resident birth-death chains (csrc/stencil_reg1d.cu): windows that
begin and end anywhere in a round of eight jumps, warps and CTAs at their
edges, against the shared-memory chain."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 13, 14, 15, 33, 419, 420, 448, 449, 840, 1700, 5040, 5041, 9001, 16001]


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("x", [0.0, 0.3, 1.0, 2.5, 7.0, 8.0, 21.0, 63.0, 150.0, 700.0])
def test_windows_across_rounds_equal_shared_memory_chain(x, prec):
    import torch
    import paper_2312_05647_gb300 as mjp
    sizes = [n for n in SIZES if prec == 1 or n < 9000]
    gen = np.random.default_rng(int(10 * x) + prec)
    theta = np.stack([gen.uniform(0.5, 1.0, len(sizes)) * np.maximum(sizes, 4) / 4.0, gen.uniform(0.5, 2.0, len(sizes))], axis=1)
    top = 1.1 * (theta[:, 0] + theta[:, 1] * np.asarray(sizes))
    t = x / top
    s0 = [int(gen.integers(0, n)) for n in sizes]
    out = {}
    for chain in (1, 2):
        b = mjp.Batch(sizes, theta, t, s0=s0, precision=prec)
        b.set_option(mjp.OPT_CHAIN, chain)
        o = b.empty_out()
        o.fill_(float("nan"))
        b.run(o)
        b.check()
        out[chain] = o.cpu().numpy()
    # The same operations in the same order.
    assert np.array_equal(out[1], out[2])


@pytest.mark.parametrize("prec", [1, 2])
def test_clusters_at_their_limits_equal_shared_memory_chain(prec):
    """Sizes at which a cluster's halo, its CTAs or the next cluster size decide."""
    import torch
    import paper_2312_05647_gb300 as mjp
    sizes = ([4913, 5039, 5040, 5041, 9823, 9824, 9825, 14700, 19647, 19649, 39296, 39400] if prec == 1
             else [3359, 3361, 6590, 6593, 9000])
    theta = np.stack([np.asarray(sizes) / 8.0, np.ones(len(sizes))], axis=1)
    t = np.linspace(20.0, 300.0, len(sizes)) / (1.1 * (theta[:, 0] + np.asarray(sizes)))
    out = {}
    for chain, halo in ((1, 0), (0, 0), (2, 32), (2, 8)):
        b = mjp.Batch(sizes, theta, t, s0=[n - 1 for n in sizes], precision=prec)
        b.set_option(mjp.OPT_CHAIN, chain)
        if halo:
            b.set_option(mjp.OPT_HALO, halo)
        o = b.empty_out()
        o.fill_(float("nan"))
        b.run(o)
        b.check()
        out[chain, halo] = o.cpu().numpy()
    for o in out.values():
        assert np.array_equal(o, out[1, 0])

"""The planner's CTA sizes (csrc/plan.cu): 8 warps up to eight observation
times, 16 above, each with a remainder of windows per warp, against the
oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
BD, TS = 1, 2


@pytest.mark.parametrize("trunc", [0, 1])
@pytest.mark.parametrize("kind,dims,th", [(BD, [70], [7.0, 0.6]), (TS, [52], [9.0, 0.7, 2.0, 1.0])])
@pytest.mark.parametrize("nt", [7, 8, 9, 16, 17, 50])
def test_loglik_of_many_windows_matches_oracle(kind, dims, th, nt, trunc):
    import paper_2312_05647_gb300 as mjp
    n = int(np.prod(dims)) * (2 if kind == TS else 1)
    gen = np.random.default_rng(nt)
    rho0 = synth.delta(n, 0)
    omega = oracle.expv(oracle.build_model(kind, dims, th), rho0, [1e-3])[1]["omega"]
    times = np.sort(gen.uniform(0.0, 250.0, nt)) / omega
    thetas = np.asarray(th) * gen.uniform(0.9, 1.1, size=(3, len(th)))
    p = oracle.expv(oracle.build_model(kind, dims, th), rho0, times)[0]
    ob = [([np.array([s])], np.array([2.0])) for s in np.argmax(p, axis=1)]  # states that carry mass at their time
    m = mjp.Model(kind, dims, th, 2)
    ll = mjp.loglik(m, mjp.Obs(n, times, ob, rho0), thetas, trunc=trunc, tol=1e-13 if trunc else 0.0)
    m.check()
    for b in range(3):
        rho = oracle.expv(oracle.build_model(kind, dims, thetas[b]), rho0, times, mode=trunc, tol=1e-13 if trunc else 0.0)[0]
        # 2 observations per time, each probability (at least 1e-2) within a
        # few hundred FP64 roundings, one per jump; the tolerance rule on either
        # side may stop a jump apart at 1e-13, 1e-11 of the probability.
        assert abs(ll[b] - oracle.loglik_from_rho(rho, ob)) <= 2 * nt * (1e-12 if not trunc else 2e-11)

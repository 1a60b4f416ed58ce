"""The FP64 SIR filter where its draws change form: probabilities near 0, 1/2 and 1, n p about the
10 that separates inversion from rejection, small and large populations; bit for bit with the
oracle's sampler."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_12973_gb300 import inputs as I

from gpu_util import rel_err, soa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npop,i0", [(3.0, 1.0), (40.0, 20.0), (1e4, 60.0), (16777216.0, 4000000.0)])
@pytest.mark.parametrize("beta,gamma", [(1e-9, 1e-9), (0.3, 0.15), (1.2, 0.6931471805599453), (5.0, 2.5), (30.0, 45.0)])
def test_fp64_draws_match_the_oracle(npop, i0, beta, gamma):
    from paper_2311_12973_gb300 import smc2 as S
    w = I.workload("sir_t30_n1024", N=2, M=160, T=6, npop=npop, i0=i0, precision=I.PREC_FP64)
    w.y = np.maximum(np.round(i0 * np.ones(6)), 1.0)
    th = np.array([[beta, gamma], [0.8 * beta, 1.1 * gamma]])
    pf = dict(pf_scheme=O.PF_SYSTEMATIC, pf_ess_frac=0.0)
    ctx = S.SMC2(S.make_config(w, ppt=2, cta_threads=96, **pf), w.y)
    ll, delta, anc = (a.cpu().numpy() for a in ctx.pf_trace(soa(th), iteration=3))
    ctx.close()
    for i in range(2):
        r_ll, r_delta, r_anc = O.pf_loglik(O.config_from(w, **pf), th[i], w.y, 3, i, trace=True)
        fin = np.isfinite(r_delta)
        assert np.array_equal(fin, np.isfinite(delta[i]))
        alive = int(fin.sum())   # a filter whose particles all die out writes no ancestors after that
        assert np.array_equal(anc[i][:alive], r_anc[:alive])
        # rounding of log-weights of up to y log y, and of the prefix sums behind them
        scale = 6 * 2 * float(np.max(w.y * np.log(np.maximum(w.y, 2.0)) + w.y))
        assert rel_err(delta[i][fin], r_delta[fin], scale) < 1e-12
        assert rel_err(ll[i], r_ll, scale) < 1e-12 if np.isfinite(r_ll) else ll[i] == r_ll

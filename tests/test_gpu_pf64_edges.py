"""The FP64 filter with up to four particles per thread at the edges of its parts: steps about the
32 whose increments are added together and about the four that share their normals, groups of
one and several warps with ragged last threads, and models outside the fixed-point range."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_12973_gb300 import inputs as I

from gpu_util import rel_err, soa

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2311_12973_gb300 import smc2
    return smc2


def _check(S, w, th, ppt, cta, **pf):
    ctx = S.SMC2(S.make_config(w, ppt=ppt, cta_threads=cta, **pf), w.y)
    ll, delta, anc = (a.cpu().numpy() for a in ctx.pf_trace(soa(th), iteration=4))
    ctx.close()
    for i in range(len(th)):
        r_ll, r_delta, r_anc = O.pf_loglik(O.config_from(w, **pf), th[i], w.y, 4, i, trace=True)
        assert np.array_equal(anc[i], r_anc), f"filter {i}: ancestors differ"
        fin = np.isfinite(r_delta)
        assert np.array_equal(fin, np.isfinite(delta[i]))
        # rounding of T steps of log-weights of this size
        scale = w.T * max(10.0, float(np.max(np.abs(r_delta[fin]), initial=0.0)))
        assert rel_err(delta[i][fin], r_delta[fin], scale) < 1e-12
        if np.isfinite(r_ll):
            assert rel_err(ll[i], r_ll, scale) < 1e-12
        else:
            assert ll[i] == r_ll


@pytest.mark.parametrize("paper", [False, True])
@pytest.mark.parametrize("T,M,ppt", [(1, 33, 1), (4, 31, 2), (5, 129, 4), (31, 64, 2), (32, 128, 4), (33, 257, 4),
                                     (65, 1, 1), (64, 500, 1)])
def test_step_and_group_edges(S, T, M, ppt, paper):
    pf = dict(pf_scheme=O.PF_MULTINOMIAL, pf_ess_frac=0.5) if paper else {}
    w = I.workload("lg_t50_n64", M=M, N=5, T=T)
    th = I.theta_near_prior(w, 5, seed=T + M, spread=0.3)
    cta = 32 * -(-M // (32 * ppt))
    _check(S, w, th, ppt, cta, **pf)


@pytest.mark.parametrize("case", ["far_observations", "large_kappa", "large_log_beta", "three_substeps"])
def test_seir_outside_the_fixed_point_range(S, case):
    w = I.workload("seir_t100_n1024", M=96, N=3, T=12, precision=I.PREC_FP64, n_sub=3 if case == "three_substeps" else 2)
    th = np.tile(np.asarray(w.prior_mean), (3, 1)) + 0.1 * np.random.default_rng(7).standard_normal((3, 4))
    if case == "far_observations":   # lambda / y above 64 and below 2^-60 within a filter
        w.y[3:6] = 1.0
        w.y[8] = 1e17
    elif case == "large_kappa":
        th[:, 2] = 15.0
    elif case == "large_log_beta":
        th[:, 0] = 33.0
    _check(S, w, th, 2, 64)

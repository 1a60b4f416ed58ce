"""The allocation-free entry point takes SEIR constants that a context refuses.  With e0 + i0 > npop the
susceptible compartment starts below zero, where the FP64 filter's fixed-point day does not hold: the
log-likelihoods are those of the plain FP64 formula (the oracle's)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2311_12973_gb300 import inputs as I

from gpu_util import rel_err, soa

pytestmark = pytest.mark.gpu

CONSTANTS = [dict(npop=100.0, e0=60.0, i0=60.0), dict(npop=1000.0, e0=900.0, i0=200.0),
             dict(npop=1000.0, e0=1000.0, i0=1e-3)]


@pytest.mark.parametrize("ppt", [1, 2, 4, 8])
@pytest.mark.parametrize("constants", CONSTANTS, ids=["small", "large", "barely"])
def test_fp64_seir_with_susceptibles_outside_the_population(constants, ppt):
    from paper_2311_12973_gb300 import smc2 as S
    w = I.workload("seir_t100_n1024", M=100, N=3, T=8, precision=I.PREC_FP64)
    th = I.theta_near_prior(w, 3, seed=3, spread=0.1)
    y = torch.tensor(w.y, dtype=torch.float64, device="cuda")
    got = S.pf_loglik_noalloc(S.make_config(w, ppt=ppt, **constants), y, soa(th), iteration=2).cpu().numpy()
    for i in range(3):
        want, delta, _ = O.pf_loglik(O.config_from(w, **constants), th[i], w.y, 2, i, trace=True)
        # rounding of T steps of log-weights of this size
        assert rel_err(got[i], want, w.T * max(10.0, float(np.max(np.abs(delta))))) < 1e-12

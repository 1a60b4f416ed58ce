"""Systematic resampling where the division in a slot's threshold is at its limits: totals up to 2^64 - 1,
the smallest and largest offsets, slot counts at powers of two and beside them, and the staged filters
(8 and 16 particles per thread), which take the same thresholds.  Exact integers throughout."""
import numpy as np
import pytest

from paper_2311_12973_gb300 import inputs as I

from gpu_util import soa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 5, 127, 128, 129, 8191, 8192, 8193, 16381, 16383, 16384])
@pytest.mark.parametrize("total", [2 ** 64 - 1, 2 ** 64 - 2, 2 ** 63, 2 ** 33 + 1, 65537])
def test_primitive(n, total):
    import torch
    from paper_2311_12973_gb300 import smc2 as S
    cuts = np.sort(np.random.default_rng(n).integers(0, total + 1, n - 1, dtype=np.uint64)) if n > 1 else []
    C = [int(c) for c in cuts] + [total]
    q = np.array([b - a for a, b in zip([0] + C[:-1], C)], dtype=np.uint64)
    upto = np.array(C, dtype=np.uint64)
    for U in (0, 2 ** 32 - 1, 0x9E3779B9):
        tau = np.array([((j << 33) + 2 * U + 1) * total // (n << 33) for j in range(n)], dtype=np.uint64)
        want = np.searchsorted(upto, tau, side="right")   # min{i : C_i > tau}
        anc = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        S.resample_systematic(torch.tensor(q.view(np.int64), device="cuda"), U, anc)
        assert np.array_equal(anc.cpu().numpy(), want)


@pytest.mark.parametrize("M", [257, 600, 1023, 1024])
def test_staged_filters_take_the_ancestors_of_the_others(M):
    import torch
    from paper_2311_12973_gb300 import smc2 as S
    w = I.workload("lg_t50_n64", N=3, M=M, T=12, precision=I.PREC_FP64)
    th = soa(I.theta_near_prior(w, 3, seed=8, spread=0.3))
    got = []
    for ppt in (2, 8, 16):
        ctx = S.SMC2(S.make_config(w, ppt=ppt, cta_threads=32 * -(-M // (32 * ppt))), w.y)
        got.append(ctx.pf_trace(th, iteration=2)[2])
        ctx.close()
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])

"""Filters of every group width from one warp to the widest, where the group's totals are formed in
different ways: ragged and whole last warps; bit for bit the same log-likelihoods from the FP32 filter
at 2, 4 and 8 particles per thread, and from the FP64 filter at 1 and 2 the same ancestors."""
import pytest

from paper_2311_12973_gb300 import inputs as I

from gpu_util import soa

pytestmark = pytest.mark.gpu

WIDTHS = [32, 33, 64, 65, 96, 97, 128, 129, 255, 256, 257, 384, 500, 512]


@pytest.mark.parametrize("model", ["lg_t50_n64", "seir_t100_n1024"])
@pytest.mark.parametrize("M", WIDTHS + [513, 1024, 1025, 2048])
def test_fp32_filter(model, M):
    import torch
    from paper_2311_12973_gb300 import smc2 as S
    w = I.workload(model, N=3, M=M, T=12, precision=I.PREC_MIXED)
    th = soa(I.theta_near_prior(w, 3, seed=6, spread=0.3))
    got = {}
    for ppt in (2, 4, 8):
        if 32 * -(-M // (32 * ppt)) > 512:
            continue
        ctx = S.SMC2(S.make_config(w, ppt=ppt, pf_family=S.PF_FP32), w.y)
        got[ppt] = ctx.pf_loglik(th, iteration=2)
        ctx.close()
    assert len(got) >= 2
    first = next(iter(got.values()))
    assert bool(torch.isfinite(first).all())
    for ll in got.values():
        assert torch.equal(ll, first)


@pytest.mark.parametrize("model", ["lg_t50_n64", "seir_t100_n1024"])
@pytest.mark.parametrize("M", WIDTHS)
def test_fp64_filter(model, M):
    import torch
    from paper_2311_12973_gb300 import smc2 as S
    w = I.workload(model, N=3, M=M, T=12, precision=I.PREC_FP64)
    th = soa(I.theta_near_prior(w, 3, seed=6, spread=0.3))
    got = []
    for ppt in (1, 2):
        threads = 32 * -(-M // (32 * ppt))
        ctx = S.SMC2(S.make_config(w, ppt=ppt, cta_threads=threads), w.y)
        got.append(ctx.pf_trace(th, iteration=2))
        ctx.close()
    assert torch.equal(got[0][2], got[1][2])
    # increments of the same weights; the thread's totals are integers, so only their logarithms' forms could differ
    assert torch.equal(got[0][1], got[1][1])

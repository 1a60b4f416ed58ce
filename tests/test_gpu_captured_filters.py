"""Filter calls captured into CUDA graphs by the caller share nothing of the context that another launch
changes: two replays on two streams, beside the context's own calls, give the values of a plain call."""
import pytest

from paper_2311_12973_gb300 import inputs as I

from gpu_util import soa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,precision,family", [("seir_t100_n1024", I.PREC_MIXED, 2), ("lg_t50_n64", I.PREC_FP64, 0)])
def test_replays_beside_one_another(name, precision, family):
    import torch
    from paper_2311_12973_gb300 import smc2 as S
    n = 8192   # several waves of work units
    w = I.workload(name, N=64, M=512, T=20, precision=precision, pf_family=family)
    stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    ctx = S.SMC2(S.make_config(w, ppt=4, cta_threads=128, pf_family=family), w.y, stream=stream)
    th = soa(I.theta_near_prior(w, n, seed=5, spread=0.3))
    torch.cuda.synchronize()
    outs = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(3)]
    want = torch.empty_like(outs[0])
    ctx.pf_loglik(th, iteration=2, out=want)
    torch.cuda.synchronize()
    graphs = [torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()]
    for g, out in zip(graphs, outs):
        with torch.cuda.graph(g, stream=stream):
            ctx.pf_loglik(th, iteration=2, out=out)
    for _ in range(3):
        for out in outs:
            out.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(other):
            graphs[0].replay()
        graphs[1].replay()                            # on the default stream
        ctx.pf_loglik(th, iteration=2, out=outs[2])   # on the context's
        torch.cuda.synchronize()
        for out in outs:
            assert torch.equal(out, want)
    ctx.close()

"""The statistics of a run of several datasets, iteration-major, below and above what the context's staging
buffer holds: the entries that smc2_get_history returns dataset by dataset."""
import numpy as np
import pytest

from paper_2311_12973_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_iter", [1, 80, 82, 120])   # 5 x 640 bytes an iteration: 256 KB lie between 81 and 82
def test_batched_statistics_equal_the_history(n_iter):
    from paper_2311_12973_gb300 import smc2 as S
    w = I.workload("lg_t50_n64", N=32, M=32, T=5, K=n_iter)
    sizes = [(32, 32, 5), (40, 32, 4), (64, 32, 3), (33, 32, 5), (32, 32, 2)]
    y = np.concatenate([w.y[:t] for _, _, t in sizes])
    ctx = S.SMC2(S.make_config(w), y, datasets=sizes)
    got = ctx.run(n_iter)
    for d in range(len(sizes)):
        hist = ctx.history(d)
        assert len(hist) == n_iter
        for row, h in zip(got, hist):
            for name, v in h.items():
                assert np.array_equal(np.asarray(row[d][name]), np.asarray(v), equal_nan=True), (d, name)
    ctx.close()

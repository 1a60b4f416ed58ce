"""Systematic resampling at the edges of the scan's runs and blocks, against the oracle bit for bit."""
import numpy as np
import pytest
import torch

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [31, 33, 511, 512, 513, 1023, 1025, 1537, 10007, 15361, 16383])
def test_run_and_block_edges(n):
    from paper_2311_12973_gb300 import smc2 as S
    rng = np.random.default_rng(n)
    for spread in (0.1, 6.0):
        q, _ = O.quantise(spread * rng.standard_normal(n))
        U = int(rng.integers(0, 2 ** 32))
        _, ref = O.systematic_from_q(q, U)
        anc = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        S.resample_systematic(torch.tensor(q.view(np.int64), device="cuda"), U, anc)
        assert np.array_equal(anc.cpu().numpy(), ref)

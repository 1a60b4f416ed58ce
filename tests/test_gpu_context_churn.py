"""Contexts made and destroyed over and over, more at once than the buffers that are kept for reuse, and from
several threads: a reused read-back buffer carries nothing over."""
import threading

import numpy as np
import pytest

from paper_2311_12973_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _run(seed, stream=None):
    from paper_2311_12973_gb300 import smc2 as S
    w = I.workload("lg_t50_n64", N=64 + 8 * (seed % 3), M=64, T=10, K=3, seed=seed)
    ctx = S.SMC2(S.make_config(w, ppt=2, cta_threads=32), w.y, stream=stream)
    stats = ctx.run(3)
    return ctx, [[s[0][k] for k in ("ess", "lse", "logz")] for s in stats], ctx.get_state(), ctx.estimate()


def _same(a, b):
    return a[1] == b[1] and all(np.array_equal(x, y) for x, y in zip(a[2] + a[3], b[2] + b[3]))


def test_more_contexts_than_kept_buffers():
    first = [_run(s) for s in range(1, 21)]
    for r in first:
        r[0].close()
    for s, r in zip(range(1, 21), first):
        again = _run(s)
        assert _same(again, r)
        again[0].close()


def test_threads_making_contexts():
    import torch
    want = {s: _run(s) for s in range(1, 9)}
    for r in want.values():
        r[0].close()
    bad = []

    def work(base):
        stream = torch.cuda.Stream()
        for n in range(24):
            s = 1 + (base + n) % 8
            r = _run(s, stream)
            if not _same(r, want[s]):
                bad.append(s)
            r[0].close()

    ts = [threading.Thread(target=work, args=(b,)) for b in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad

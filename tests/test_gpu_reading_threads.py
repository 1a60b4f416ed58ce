"""Several host threads reading one context at the same time, and beside a run: every call returns its own
values (the calls stage their copies through one buffer of the context)."""
import threading

import numpy as np
import pytest

from paper_2311_12973_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _same(a, b):
    return all(np.array_equal(np.asarray(x), np.asarray(y)) for x, y in zip(a, b))


def _in_threads(jobs):
    bad = []

    def call(job):
        try:
            job(bad)
        except Exception as e:  # a status word read from another call's bytes
            bad.append(repr(e))

    ts = [threading.Thread(target=call, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad[:3]


def test_state_and_estimate_read_together():
    from paper_2311_12973_gb300 import smc2 as S
    w = I.workload("lg_t50_n64", N=256, M=64, T=20, K=4)
    ctx = S.SMC2(S.make_config(w), w.y)
    ctx.run(4)
    state, est, hist = ctx.get_state(), ctx.estimate(), [h["lse"] for h in ctx.history()]

    def states(bad):
        bad += ["state" for _ in range(1000) if not _same(ctx.get_state(), state)]

    def estimates(bad):
        bad += ["estimate" for _ in range(1000) if not _same(ctx.estimate(), est)]

    def histories(bad):
        bad += ["history" for _ in range(300) if [h["lse"] for h in ctx.history()] != hist]

    _in_threads([states, estimates, histories, states])
    ctx.close()


def test_statistics_of_a_run_beside_readers():
    from paper_2311_12973_gb300 import smc2 as S
    w = I.workload("lg_t50_n64", N=256, M=64, T=20, K=40)
    ctx = S.SMC2(S.make_config(w), w.y)
    want = [r[0]["lse"] for r in ctx.run(40)]
    ctx.reset(w.seed)
    got, done = [], threading.Event()

    def run(bad):
        try:
            for _ in range(40):
                got.append(ctx.run(1)[0][0]["lse"])
        finally:
            done.set()

    def read(bad):
        while not done.is_set():
            ctx.get_state()
            ctx.sync()

    _in_threads([run, read, read])
    assert got == want
    ctx.close()

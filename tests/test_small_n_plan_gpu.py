"""Small-N tensor-core path: a run's trajectory does not depend on how the runs of its
context are spread over the SMs (chunk length, items per CTA, runs per group)."""
import numpy as np
import pytest

from paper_2308_02329_gb300 import chym, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,D", [(20, 1), (100, 2), (33, 3), (128, 4), (17, 5), (64, 8)])
@pytest.mark.parametrize("R", [1, 3, 609, 2432, 2433, 10007])
def test_spread_of_the_runs_leaves_states_unchanged(N, D, R):
    J = inputs.gaussian(N, 3) if D == 3 else inputs.sk_pm1(N, 3)
    ctx = chym.Context(J, D, chym.J_REAL if D == 3 else chym.J_PM1)
    prm = chym.Params(eps=0.25 if D == 3 else 0.25 / np.sqrt(N), prec=chym.PREC_BF16X2)
    sched = chym.Schedule(1, 3, 9)
    seeds = inputs.run_seeds(21, R)
    ctx.run(prm, np.array([0.8]), seeds, 7, sched)
    X, k = ctx.get_state()
    assert k == 7
    # the last runs again, alone: 5 runs take other CTAs, groups and chunks
    few = min(R, 5)
    ctx.run(prm, np.array([0.8]), seeds[R - few:], 7, sched)
    Y, _ = ctx.get_state()
    assert np.array_equal(X[R - few:], Y)
    # and all of them as a batch
    ctx.run(prm, np.array([0.8]), seeds, 0, sched)
    b = chym.Batch([ctx])
    b.run([prm], [sched], 7)
    b.status()
    assert np.array_equal(ctx.get_state()[0], X)
    b.close()
    ctx.close()


# runs per context: CTAs shared between contexts, whole CTAs for each, one run, more contexts than SMs
@pytest.mark.parametrize("D,runs", [(3, [228] * 5), (2, [105, 105, 105]), (4, [1, 300, 7]), (3, [4096, 5]),
                                    (1, [3] * 160), (8, [45, 999, 2])])
def test_spread_of_several_contexts_leaves_states_unchanged(D, runs):
    sched = chym.Schedule(1, 3, 9)
    prm = chym.Params(eps=0.06, prec=chym.PREC_BF16X2)
    ctxs, alone = [], []
    for i, R in enumerate(runs):
        ctx = chym.Context(inputs.sk_pm1(18 + i % 7, 3 + i), D, chym.J_PM1)
        seeds = inputs.run_seeds(50 + i, R)
        ctx.run(prm, np.array([0.8]), seeds, 7, sched)
        alone.append(ctx.get_state()[0])
        ctx.run(prm, np.array([0.8]), seeds, 0, sched)
        ctxs.append(ctx)
    b = chym.Batch(ctxs)
    b.run([prm] * len(runs), [sched] * len(runs), 7)
    b.status()
    for ctx, X in zip(ctxs, alone):
        assert np.array_equal(ctx.get_state()[0], X)
    b.close()
    for ctx in ctxs:
        ctx.close()


@pytest.mark.parametrize("D,R", [(1, 300), (2, 700), (3, 512), (3, 1216), (4, 512), (5, 512), (6, 500), (8, 600)])
def test_calls_on_several_streams_share_the_sms(D, R):
    """Eight contexts on streams of their own, few runs an SM each: states as alone, and where
    two CTAs fit an SM the calls do not queue for whole SMs."""
    torch = pytest.importorskip("torch")
    import time
    n, steps = 8, 800
    sched = chym.Schedule(1, 300, 600)
    ctxs, prm, seeds, alone, streams = [], [], [], [], []
    for i in range(n):
        real = i % 3 == 2
        J = inputs.gaussian(100, 3 + i) if real else inputs.sk_pm1(100 - 7 * i, 3 + i)
        ctx = chym.Context(J, D, chym.J_REAL if real else chym.J_PM1)
        ctxs.append(ctx)
        prm.append(chym.Params(eps=0.25 if real else 0.025, prec=chym.PREC_BF16X2))
        seeds.append(inputs.run_seeds(60 + i, R))
        ctx.run(prm[i], np.array([0.8]), seeds[i], steps, sched)
        alone.append(ctx.get_state()[0])
        streams.append(torch.cuda.Stream())

    def seconds(which):
        for i in which:
            ctxs[i].run(prm[i], np.array([0.8]), seeds[i], 0, sched)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for i in which:
            ctxs[i].run(prm[i], None, None, steps, sched, streams[i].cuda_stream)
        torch.cuda.synchronize()
        return time.perf_counter() - t0

    one = min(max(seconds([i]) for i in (0, 2)) for _ in range(3))
    t = min(seconds(range(n)) for _ in range(3))
    for ctx, X in zip(ctxs, alone):
        assert np.array_equal(ctx.get_state()[0], X)
    if D == 3 and R == 512:
        assert t < 5.5 * one, (t, one)
    for ctx in ctxs:
        ctx.close()

"""Plain FP32 form: a run's trajectory does not depend on how many runs a thread and a block
take (both shrink with the number of runs)."""
import numpy as np
import pytest

from paper_2308_02329_gb300 import chym, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", ["sk", "mobius"])
@pytest.mark.parametrize("D,R", [(1, 40001), (1, 12000), (2, 20003), (2, 7000), (3, 20000), (3, 6001), (4, 20001),
                                 (4, 6000), (5, 10007), (7, 601), (8, 10000)])
def test_runs_per_thread_leave_states_unchanged(D, R, graph):
    N = 41 if graph == "sk" else 42
    J = inputs.sk_pm1(N, 3) if graph == "sk" else inputs.mobius_ladder(N)
    ctx = chym.Context(J, D)
    prm = chym.Params(eps=0.04, prec=chym.PREC_FP32)
    sched = chym.Schedule(1, 3, 8)
    seeds = inputs.run_seeds(5, R)
    h = np.array([0.8])
    ctx.run(prm, h, seeds, 6, sched)
    X, _ = ctx.get_state()
    for lo in (0, R // 2, R - 5):
        ctx.run(prm, h, seeds[lo:lo + 5], 6, sched)
        assert np.array_equal(ctx.get_state()[0], X[lo:lo + 5])
    ctx.close()

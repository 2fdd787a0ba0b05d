"""FP64 form against the oracle where its split of the work has edges: several runs per block
with a ragged last one, odd N D (noise pairs across spins), one or two Philox blocks per
spin, sparse rows, more values than threads, buffers beyond shared memory."""
import numpy as np
import pytest

import oracle.oracle as O
from paper_2308_02329_gb300 import chym, inputs
from tests.helpers import make_case, oracle_params, oracle_schedule, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,D,n_h,reps,graph", [
    (1, 1, 1, 2, "sk"), (7, 1, 2, 200, "sk"), (9, 2, 1, 307, "gauss"), (20, 3, 8, 61, "sk"),
    (5, 4, 1, 1601, "sk"), (13, 5, 3, 120, "sk"), (40, 6, 2, 90, "gauss"), (33, 7, 1, 155, "sk"),
    (25, 8, 2, 160, "sk"), (100, 4, 1, 311, "mobius"), (301, 2, 1, 5, "mobius"), (1300, 8, 1, 2, "gauss")])
def test_state_matches_oracle(N, D, n_h, reps, graph):
    if graph == "mobius":
        N += N % 2
    J, eps, h, seeds = make_case(N, D, n_h, reps, 23, graph)
    ctx = chym.Context(J, D, chym.J_REAL if graph == "gauss" else chym.J_PM1)
    prm = chym.Params(eps=eps, prec=chym.PREC_FP64)
    steps = 12 if N < 1000 else 3
    sch = chym.Schedule(1, steps // 3, steps - 1)   # ramp and its end inside the run
    ctx.run(prm, h, seeds, steps, sch)
    X, k = ctx.get_state()
    assert k == steps
    Xo = O.run(J, D, inputs.h_per_run(h, reps), seeds, oracle_params(prm), oracle_schedule(sch), steps)
    assert rel_err(X, Xo) <= 1e-10   # FP64 mode, as in the other parity tests
    ctx.close()


@pytest.mark.parametrize("N,D,n_h,reps,graph", [
    (160, 3, 2, 15, "sk"), (20, 3, 7, 200, "sk"), (100, 2, 1, 1201, "mobius"), (300, 1, 1, 41, "gauss"),
    (130, 8, 3, 7, "sk"), (40, 6, 2, 401, "gauss"), (200, 3, 1, 305, "gauss"), (128, 5, 1, 153, "mobius"),
    (64, 4, 1, 153, "sk"), (600, 2, 1, 3, "mobius"), (1100, 4, 1, 2, "sk"), (21, 7, 1, 1000, "sk"), (20, 8, 1, 607, "sk")])
def test_full_warps_one_cta_an_sm(N, D, n_h, reps, graph):
    """Sizes whose (run, spin) slots fill the warps of one block per SM: several runs per block
    with a ragged last one, slots from 80 (D = 8), just above 128 and above 512, J in and beyond shared memory,
    sparse rows, one component."""
    test_state_matches_oracle(N, D, n_h, reps, graph)


@pytest.mark.parametrize("N,D,n_h,reps,graph", [
    (10, 3, 1, 9800, "sk"), (20, 3, 1, 4096, "sk"), (100, 2, 1, 4097, "sk"), (48, 4, 1, 9733, "mobius"),
    (101, 8, 1, 1530, "gauss"), (300, 3, 1, 256, "sk"), (500, 3, 1, 1369, "mobius"), (300, 1, 1, 7904, "mobius")])
def test_several_waves(N, D, n_h, reps, graph):
    """More runs than one block per SM holds, and blocks of half the runs where one would leave
    most of a pass idle: equal waves, the last one ragged."""
    test_state_matches_oracle(N, D, n_h, reps, graph)


def test_two_waves_take_no_longer_than_twice_one():
    torch = pytest.importorskip("torch")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctx = chym.Context(inputs.sk_pm1(100, 3), 3)
    prm, sch = chym.Params(eps=0.025, prec=chym.PREC_FP64), chym.Schedule(1, 100, 200)

    def ms(R):
        ctx.run(prm, np.array([0.8]), inputs.run_seeds(4, R), 0, sch)
        best = np.inf
        for _ in range(4):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            ctx.run(prm, None, None, 20, sch, torch.cuda.current_stream().cuda_stream)
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1))
        return best

    assert ms(52 * sms) < 2.1 * ms(26 * sms)   # 26 runs fill a block's shared memory
    ctx.close()

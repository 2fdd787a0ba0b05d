"""FP32 form over the compressed rows of large sparse graphs against the oracle: rows longer than
the nonzeros held in registers and empty ones, every Philox block layout, several runs per
block with a ragged last one, weights, a ramp that ends inside the run, odd first steps."""
import numpy as np
import pytest

import oracle.oracle as O
from paper_2308_02329_gb300 import chym, inputs
from tests.helpers import oracle_params, oracle_schedule, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,D,R,density", [
    (2501, 1, 309, 0.003), (2000, 2, 160, 0.002), (1024, 3, 5, 0.0), (1501, 3, 457, 0.004), (1300, 4, 153, 0.01),
    (901, 5, 7, 0.01), (1100, 8, 3, 0.004)])
@pytest.mark.parametrize("weighted", [False, True])
def test_state_matches_oracle(N, D, R, density, weighted):
    J = inputs.sparse_pm1(N, density, 9)
    ctx = chym.Context(J, D)
    w = np.linspace(0.5, 1.5, N) if weighted else np.ones(N)
    if weighted:
        ctx.set_coupling_weights(w)
    prm = chym.Params(eps=0.1, prec=chym.PREC_FP32)
    assert ctx.uses_csr(chym.PREC_FP32)
    sch = chym.Schedule(1, 3, 10)
    h = np.array([0.7])
    seeds = inputs.run_seeds(31, R)
    ctx.run(prm, h, seeds, 5, sch)
    ctx.run(prm, None, None, 7, sch)      # continues at an odd step
    X, k = ctx.get_state()
    assert k == 12
    few = np.unique(np.linspace(0, R - 1, min(R, 6)).astype(int))
    Xo = O.run(np.diag(w) @ J, D, np.full(len(few), 0.7), seeds[few], oracle_params(prm), oracle_schedule(sch), 12)
    assert rel_err(X[few], Xo) <= 1e-4    # FP32 mode over a short horizon, as in the other parity tests
    ctx.close()

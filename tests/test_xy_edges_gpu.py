"""Best-axis readout against the oracle around the switch from a warp to a block per run, with
equal angles and diverged runs; and, with a spin of zero length (it keeps +1, so that opposite
axes differ), against the documented turn of the axis written out in numpy."""
import math

import numpy as np
import pytest

import oracle.oracle as O
from paper_2308_02329_gb300 import chym, inputs

pytestmark = pytest.mark.gpu


def _turn(J, x):
    """Lowest energy as the axis turns from inside the interval that wraps through pi."""
    key = {}
    for p, (a, b) in enumerate(x):
        if a != 0 or b != 0:
            k = math.fmod(math.atan2(b, a) + 0.5 * math.pi, math.pi)
            key[p] = k + math.pi if k < 0 else k
    order = sorted(key, key=lambda p: (key[p], p))
    phi = 0.5 * (key[order[-1]] + key[order[0]] + math.pi) if order else 0.0
    s = np.where(x[:, 0] * math.cos(phi) + x[:, 1] * math.sin(phi) >= 0, 1.0, -1.0)
    best = -(s @ J @ s)
    for i, p in enumerate(order):
        s[p] = -s[p]
        if i + 1 == len(order) or key[order[i + 1]] != key[p]:
            best = min(best, -(s @ J @ s))
    return best


@pytest.mark.parametrize("prec", [chym.PREC_FP32, chym.PREC_FP64])
@pytest.mark.parametrize("N,R,graph", [(1, 3, "sk"), (2, 9, "sk"), (32, 8, "sparse"), (33, 17, "sk"), (100, 5, "sparse"),
                                       (255, 4, "sk"), (256, 9, "sk"), (257, 3, "sk"), (300, 2, "sparse")])
def test_best_axis_matches_oracle(N, R, graph, prec):
    J = inputs.sk_pm1(N, 8) if graph == "sk" else inputs.sparse_pm1(N, 0.2, 8)
    ctx = chym.Context(J, 2)
    rng = np.random.default_rng(4)
    X = rng.standard_normal((R, N, 2)).astype(np.float32).astype(np.float64)
    X[0, 0] = 0.0                                  # never flips
    X[R - 1, N // 2:] = X[R - 1, N // 2]           # equal angles flip together
    if R > 4:
        X[1, N - 1, 1] = np.inf
    ctx.set_state(X, np.ones(1), np.arange(R, dtype=np.uint64), 0, prec)
    E, S = ctx.readout_xy(spins=True)
    s = chym.unpack_spins(S, N).astype(np.float64)
    for r in range(R):
        if R > 4 and r == 1:
            assert np.isnan(E[r])
            continue
        assert E[r] == (_turn(J, X[r]) if r == 0 else O.round_xy(J, X[r])[0])
        assert E[r] == -(s[r] @ J @ s[r])
    ctx.close()

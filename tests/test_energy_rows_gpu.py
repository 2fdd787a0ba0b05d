"""Ising energies, packed spins and segment energies against plain numpy on the returned
state, at the edges of the energy kernels: spin-word boundaries, run counts on both sides
of the switch between few and many runs per block, +-1 and real couplings."""
import numpy as np
import pytest

from paper_2308_02329_gb300 import chym, inputs

pytestmark = pytest.mark.gpu


def _state(ctx, N, D, R, prec, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((R, N, D)).astype(np.float32).astype(np.float64)
    X[0, 0, 0] = 0.0                       # a tie reads +1
    if R > 2:
        X[1, N - 1, D - 1] = np.inf        # diverged runs read NaN
        X[2, 0, 0] = np.nan
    ctx.set_state(X, np.ones(1), np.arange(R, dtype=np.uint64), 0, prec)
    return X


def _field_energy(J, s):
    return -np.einsum("rp,pq,rq->r", s, J, s)


@pytest.mark.parametrize("kind", ["pm1", "real", "wide"])
@pytest.mark.parametrize("N,D,R,prec", [
    (1, 1, 1, chym.PREC_FP32), (2, 3, 5, chym.PREC_FP64), (63, 2, 9, chym.PREC_FP32),
    (64, 1, 17, chym.PREC_BF16X2), (65, 4, 3, chym.PREC_FP64), (129, 3, 2431, chym.PREC_FP32),
    (100, 2, 2433, chym.PREC_BF16X2), (67, 1, 4863, chym.PREC_FP32), (70, 2, 4865, chym.PREC_FP64),
    (1030, 1, 6, chym.PREC_FP32)])
def test_energies_match_numpy(kind, N, D, R, prec):
    J = inputs.sk_pm1(N, 5) if kind == "pm1" else inputs.gaussian(N, 5)
    if kind == "wide":                     # rows of very different scale
        sc = 10.0 ** np.linspace(-60, 60, N)
        J = J * np.sqrt(np.outer(sc, sc))
        J = np.triu(J, 1) + np.triu(J, 1).T
    ctx = chym.Context(J, D, chym.J_PM1 if kind == "pm1" else chym.J_REAL)
    X = _state(ctx, N, D, R, prec, 11)
    E, S = ctx.energy(spins=True)
    s = np.where(X[..., 0] >= 0, 1.0, -1.0)
    ok = np.isfinite(X).all(axis=(1, 2))
    assert np.array_equal(np.isfinite(E), ok)
    assert np.array_equal(chym.unpack_spins(S, N)[ok], s[ok])
    want = _field_energy(J, s)
    if kind == "pm1":
        assert np.array_equal(E[ok], want[ok])
    else:
        # rounding of each row's exact local field and of the sum over rows: N terms, each
        # partial sum below sum |J|; numpy's own N^2-term sum allowed for as much again
        tol = 4 * N * 2.0 ** -53 * np.abs(J).sum()
        assert np.max(np.abs(E[ok] - want[ok])) <= tol
    ctx.close()


@pytest.mark.parametrize("kind", ["pm1", "real"])
@pytest.mark.parametrize("N,D,R,cuts", [
    (5, 1, 3, [0, 5]), (64, 2, 9, [0, 1, 63, 64]), (128, 2, 40, [0, 10, 64, 65, 100, 128]),
    (130, 1, 2433, [0, 63, 129, 130]), (200, 3, 7, [0, 120, 200]), (128, 1, 5, list(range(129)))])
def test_segment_energies_match_numpy(kind, N, D, R, cuts):
    J = np.zeros((N, N))
    for i, (a, b) in enumerate(zip(cuts[:-1], cuts[1:])):
        J[a:b, a:b] = inputs.sk_pm1(b - a, i) if kind == "pm1" else inputs.gaussian(b - a, i)
    if kind == "pm1":                      # couplings across segments do not count
        J[0, N - 1] = J[N - 1, 0] = 1.0 if len(cuts) > 2 else J[0, N - 1]
    ctx = chym.Context(J, D, chym.J_PM1 if kind == "pm1" else chym.J_REAL)
    X = _state(ctx, N, D, R, chym.PREC_FP32, 12)
    E = ctx.energy_segments(cuts)
    s = np.where(X[..., 0] >= 0, 1.0, -1.0)
    fin = np.isfinite(X).all(axis=2)
    for i, (a, b) in enumerate(zip(cuts[:-1], cuts[1:])):
        ok = fin[:, a:b].all(axis=1)
        assert np.array_equal(np.isfinite(E[:, i]), ok)
        want = _field_energy(J[a:b, a:b], s[:, a:b])
        tol = 0.0 if kind == "pm1" else 4 * (b - a) * 2.0 ** -53 * np.abs(J[a:b, a:b]).sum()
        assert np.max(np.abs(E[ok, i] - want[ok]), initial=0.0) <= tol
    ctx.close()


@pytest.mark.parametrize("N,R,prec", [(511, 9, chym.PREC_FP32), (512, 1, chym.PREC_FP64), (513, 65, chym.PREC_FP32),
                                      (1500, 64, chym.PREC_FP8), (777, 1215, chym.PREC_FP32)])
def test_rows_shared_between_blocks(N, R, prec):
    """Few runs of a large +-1 J: the rows of a run are split over several blocks."""
    J = inputs.sk_pm1(N, 5)
    ctx = chym.Context(J, 2, chym.J_PM1)
    X = _state(ctx, N, 2, R, prec, 13)
    E, S = ctx.energy(spins=True)
    s = np.where(X[..., 0] >= 0, 1.0, -1.0)
    ok = np.isfinite(X).all(axis=(1, 2))
    assert np.array_equal(np.isfinite(E), ok)
    assert np.array_equal(chym.unpack_spins(S, N)[ok], s[ok])
    assert np.array_equal(E[ok], _field_energy(J, s)[ok])
    ctx.close()


def test_real_couplings_device_memory():
    """A context with real couplings holds them in FP64, FP32 (twice, one with padded rows) and
    the digit planes of the tiles on and above the diagonal: 23 bytes an entry."""
    torch = pytest.importorskip("torch")
    N = 2048
    J = inputs.gaussian(N, 5)
    chym.Context(inputs.gaussian(16, 5), 1, chym.J_REAL).close()   # the module's own memory
    free = torch.cuda.mem_get_info()[0]
    ctx = chym.Context(J, 1, chym.J_REAL)
    used = free - torch.cuda.mem_get_info()[0]
    assert used <= 25 * N * N
    ctx.close()

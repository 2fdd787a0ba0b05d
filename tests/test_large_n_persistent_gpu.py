"""Large-N tensor-core path: a run's trajectory depends neither on the column tiles, lists and
phases its context's work is cut into, nor on the launches a call is cut into, nor on how
many SMs the persistent launch finds free."""
import numpy as np
import pytest

from paper_2308_02329_gb300 import chym, inputs

pytestmark = pytest.mark.gpu


def _ctx(N, D, kind):
    J = inputs.gaussian(N, 3) if kind == "gauss" else inputs.sk_pm1(N, 3)
    ctx = chym.Context(J, D, chym.J_REAL if kind == "gauss" else chym.J_PM1)
    eps = 0.25 if kind == "gauss" else 0.25 / np.sqrt(N)
    return ctx, eps


def _states(ctx, prm, sched, seeds, steps, stream=0):
    ctx.run(prm, np.array([0.8]), seeds, steps, sched, stream)
    X, k = ctx.get_state(stream)
    assert k == steps
    return X


@pytest.mark.parametrize("N,D,kind,prec", [
    (129, 1, "sk", chym.PREC_BF16X2), (256, 2, "sk", chym.PREC_FP8), (257, 3, "gauss", chym.PREC_BF16X2),
    (385, 4, "sk", chym.PREC_FP8), (200, 5, "gauss", chym.PREC_BF16X2), (130, 8, "sk", chym.PREC_FP8)])
@pytest.mark.parametrize("R", [1, 9, 24, 100, 130, 1030])
def test_tiling_leaves_states_unchanged(N, D, kind, prec, R):
    ctx, eps = _ctx(N, D, kind)
    prm = chym.Params(eps=eps, prec=prec)
    sched = chym.Schedule(1, 3, 8)
    seeds = inputs.run_seeds(5, R)
    X = _states(ctx, prm, sched, seeds, 6)
    few = min(R, 5)   # the last runs alone: other tiles, widths and lists
    assert np.array_equal(X[R - few:], _states(ctx, prm, sched, seeds[R - few:], 6))
    ctx.close()


@pytest.mark.parametrize("D,R", [(8, 9760), (4, 19500)])
def test_phases_leave_states_unchanged(D, R):
    """More tiles than four per SM and enough steps: the column tiles advance in phases."""
    ctx, eps = _ctx(130, D, "sk")
    prm = chym.Params(eps=eps, prec=chym.PREC_BF16X2)
    sched = chym.Schedule(1, 16, 33)
    seeds = inputs.run_seeds(6, R)
    X = _states(ctx, prm, sched, seeds, 33)
    for lo in (0, R // 2, R - 64):
        assert np.array_equal(X[lo:lo + 64], _states(ctx, prm, sched, seeds[lo:lo + 64], 33))
    ctx.close()


def test_launch_boundaries_leave_states_unchanged():
    """2060 steps take three launches; two calls cut them elsewhere."""
    ctx, eps = _ctx(140, 3, "sk")
    prm = chym.Params(eps=eps, prec=chym.PREC_FP8)
    sched = chym.Schedule(1, 1000, 2060)
    seeds = inputs.run_seeds(7, 40)
    X = _states(ctx, prm, sched, seeds, 2060)
    ctx.run(prm, np.array([0.8]), seeds, 777, sched)
    ctx.run(prm, None, None, 2060 - 777, sched)
    assert np.array_equal(ctx.get_state()[0], X)
    ctx.close()


@pytest.mark.parametrize("busy_runs", [40, 300, 590])
def test_fewer_free_sms_leave_states_unchanged(busy_runs):
    """Another stream's persistent small-N launch holds some SMs while the large-N one starts."""
    torch = pytest.importorskip("torch")
    ctx, eps = _ctx(260, 4, "sk")
    prm = chym.Params(eps=eps, prec=chym.PREC_BF16X2)
    sched = chym.Schedule(1, 5, 20)
    seeds = inputs.run_seeds(8, 4096)
    X = _states(ctx, prm, sched, seeds, 15)
    small, seps = _ctx(100, 4, "sk")
    sprm = chym.Params(eps=seps, prec=chym.PREC_BF16X2)
    ssched, sseeds = chym.Schedule(1, 10000, 20000), inputs.run_seeds(9, busy_runs)
    S = _states(small, sprm, ssched, sseeds, 20000)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    small.run(sprm, np.array([0.8]), sseeds, 20000, ssched, a.cuda_stream)
    ctx.run(prm, np.array([0.8]), seeds, 15, sched, b.cuda_stream)
    assert np.array_equal(ctx.get_state(b.cuda_stream)[0], X)
    assert np.array_equal(small.get_state(a.cuda_stream)[0], S)
    small.close()
    ctx.close()


@pytest.mark.parametrize("D,wide,narrow", [(4, 64, 32), (2, 128, 32), (1, 256, 32)])
def test_wide_and_narrow_tiles_in_one_list(D, wide, narrow):
    """Tiles of wide and of narrow columns in turn, M tiles with two live rows, several a CTA:
    the epilogue's warps finish far apart, and a tile counts as finished only when all have."""
    # a launch has at least 152 tiles, so a CTA's list holds wide and narrow ones
    sizes = [(130, 160 * wide), (130, 16), (200, 9), (130, 33), (257, 5), (130, narrow), (140, 1), (385, 16)]
    prm, sched = [], chym.Schedule(1, 40, 200)
    ctxs, alone, seeds = [], [], []
    for i, (N, R) in enumerate(sizes):
        ctx, eps = _ctx(N, D, "sk" if i % 2 else "gauss")
        ctxs.append(ctx)
        prm.append(chym.Params(eps=eps, prec=chym.PREC_BF16X2))
        seeds.append(inputs.run_seeds(20 + i, R))
        alone.append(_states(ctx, prm[-1], sched, seeds[-1], 200))
    batch = chym.Batch(ctxs)
    batch.set_shapes({"rt": [wide if d == D else 0 for d in range(1, 9)]})
    for i, ctx in enumerate(ctxs):
        ctx.run(prm[i], np.array([0.8]), seeds[i], 0, sched)
    batch.run(prm, [sched] * len(ctxs), 200)
    batch.status()
    for ctx, X in zip(ctxs, alone):
        assert np.array_equal(ctx.get_state()[0], X)
    batch.close()
    for ctx in ctxs:
        ctx.close()


def test_short_tiles_in_long_walks():
    """Thousands of the shortest tiles a CTA: the publisher stays within two tiles of the
    epilogue whatever their times, and no wait runs out."""
    sched, n, steps = chym.Schedule(1, 400, 1100), 220, 1100
    ctxs, prm, seeds = [], [], []
    for i in range(n):
        ctx, eps = _ctx(129 + i % 3, 1, "sk")
        ctxs.append(ctx)
        prm.append(chym.Params(eps=eps, prec=chym.PREC_FP8))
        seeds.append(inputs.run_seeds(50 + i, 1 + i % 9))
        ctx.run(prm[i], np.array([0.8]), seeds[i], 0, sched)
    batch = chym.Batch(ctxs)
    batch.run(prm, [sched] * n, steps)
    batch.status()
    got = {i: ctxs[i].get_state()[0] for i in (0, 1, 100, 219)}
    for i, X in got.items():
        assert np.array_equal(X, _states(ctxs[i], prm[i], sched, seeds[i], steps))
    batch.close()
    for ctx in ctxs:
        ctx.close()


def _dims_batch(specs, steps, sched):
    """Contexts (N, D, R) with a state each, and the batch over them."""
    ctxs, prm, seeds = [], [], []
    for i, (N, D, R) in enumerate(specs):
        ctx, eps = _ctx(N, D, "gauss" if i % 3 == 2 else "sk")
        ctxs.append(ctx)
        prm.append(chym.Params(eps=eps, prec=chym.PREC_FP8 if i % 2 else chym.PREC_BF16X2))
        seeds.append(inputs.run_seeds(70 + i, R))
        ctx.run(prm[i], np.array([0.8]), seeds[i], 0, sched)
    return ctxs, prm, seeds, chym.Batch(ctxs)


@pytest.mark.parametrize("specs", [
    [(130, 4, 9800), (300, 4, 700), (520, 4, 33), (200, 4, 2500)],                       # one D, phases
    [(260, 2, 9000), (260, 3, 6000), (200, 2, 40), (390, 8, 3000), (150, 3, 5), (640, 8, 100)],  # in turn
    [(260, 1, 500), (390, 4, 300), (640, 6, 64), (520, 4, 16), (130, 7, 9)]])              # side by side
def test_phases_of_several_contexts_and_dims(specs):
    sched = chym.Schedule(1, 30, 70)
    ctxs, prm, seeds, batch = _dims_batch(specs, 70, sched)
    batch.run(prm, [sched] * len(ctxs), 70)
    batch.status()
    got = [ctx.get_state()[0] for ctx in ctxs]
    for ctx, p, sd, X in zip(ctxs, prm, seeds, got):
        assert np.array_equal(X, _states(ctx, p, sched, sd, 70))
    batch.close()
    for ctx in ctxs:
        ctx.close()


def test_several_dims_take_no_longer_than_one_after_the_other():
    """Many uneven instances of four D in one batch against the four batches of one D each."""
    torch = pytest.importorskip("torch")
    sched, steps = chym.Schedule(1, 1000, 2000), 200
    rng = np.random.default_rng(4)
    specs = [(int(rng.integers(250, 1100)), (2, 3, 4, 8)[i % 4], 64) for i in range(200)]
    ctxs, prm, _, batch = _dims_batch(specs, 0, sched)
    parts = [(batch, list(range(len(specs))))]
    for D in (2, 3, 4, 8):
        of = [i for i, s in enumerate(specs) if s[1] == D]
        parts.append((chym.Batch([ctxs[i] for i in of]), of))

    def ms(b, of):
        best = np.inf
        for rep in range(4):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            b.run([prm[i] for i in of], [sched] * len(of), steps, torch.cuda.current_stream().cuda_stream)
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1)) if rep else best
        b.status()
        return best

    t = [ms(*p) for p in parts]
    assert t[0] < 1.15 * sum(t[1:]), t
    for b, _ in parts:
        b.close()
    for ctx in ctxs:
        ctx.close()


@pytest.mark.parametrize("busy_steps", [(1500,), (600, 1200, 2400, 4800)])
def test_sms_that_become_free_are_taken(busy_steps):
    """Small-N runs of other streams hold most SMs for the first few ms of a large-N call: it
    stops and goes on where it stopped, on all SMs, and takes little longer than they do."""
    torch = pytest.importorskip("torch")
    import time
    ctx, eps = _ctx(520, 4, "sk")
    prm = chym.Params(eps=eps, prec=chym.PREC_FP8)
    steps, sched = 1501, chym.Schedule(1, 700, 1400)
    seeds = inputs.run_seeds(8, 4096)
    X = _states(ctx, prm, sched, seeds, steps)
    small, ssched = [], chym.Schedule(1, 10000, 20000)
    for i, n in enumerate(busy_steps):   # 140 CTAs of four runs in all
        c, seps = _ctx(100, 4, "sk")
        small.append((c, chym.Params(eps=seps, prec=chym.PREC_BF16X2), inputs.run_seeds(9 + i, 560 // len(busy_steps)), n,
                      torch.cuda.Stream()))
        c.run(small[-1][1], np.array([0.8]), small[-1][2], 10, ssched)
    own = torch.cuda.Stream()

    def seconds(beside):
        ctx.run(prm, np.array([0.8]), seeds, 0, sched, own.cuda_stream)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        if beside:
            for c, p, _, n, stream in small:
                c.run(p, None, None, n, ssched, stream.cuda_stream)
            time.sleep(2e-4)
        if beside != "only":
            ctx.run(prm, None, None, steps, sched, own.cuda_stream)
        torch.cuda.synchronize()
        return time.perf_counter() - t0

    alone = min(seconds(False) for _ in range(3))
    assert np.array_equal(ctx.get_state()[0], X)
    busy = min(seconds("only") for _ in range(3))
    t = []
    for _ in range(3):
        t.append(seconds(True))
        assert np.array_equal(ctx.get_state()[0], X)
    assert min(t) < 2.0 * alone + busy, (t, alone, busy)
    for c in small:
        c[0].close()
    ctx.close()


@pytest.mark.parametrize("N,D,R,kind", [(250, 3, 1024, "gauss"), (260, 4, 1200, "sk"), (130, 8, 1000, "sk"), (520, 4, 8192, "sk")])
@pytest.mark.parametrize("busy_runs", [304, 600])
def test_late_ctas_and_narrow_tiles_or_phases(N, D, R, kind, busy_runs):
    """16- and 24-run tiles, several a CTA while SMs are held elsewhere, and phases once they are free."""
    torch = pytest.importorskip("torch")
    ctx, eps = _ctx(N, D, kind)
    prm = chym.Params(eps=eps, prec=chym.PREC_BF16X2)
    steps, sched = 450, chym.Schedule(1, 200, 400)
    seeds = inputs.run_seeds(8, R)
    X = _states(ctx, prm, sched, seeds, steps)
    small, seps = _ctx(100, 4, "sk")
    sprm, ssched = chym.Params(eps=seps, prec=chym.PREC_BF16X2), chym.Schedule(1, 10000, 20000)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    ctx.run(prm, np.array([0.8]), seeds, 0, sched, b.cuda_stream)
    small.run(sprm, np.array([0.8]), inputs.run_seeds(9, busy_runs), 0, ssched, a.cuda_stream)
    torch.cuda.synchronize()
    small.run(sprm, None, None, 700, ssched, a.cuda_stream)   # about a millisecond
    ctx.run(prm, None, None, steps, sched, b.cuda_stream)
    assert np.array_equal(ctx.get_state(b.cuda_stream)[0], X)
    small.close()
    ctx.close()


@pytest.mark.parametrize("other", [(100, 3, 1024, "sk", chym.PREC_FP64), (100, 4, 4096, "sk", chym.PREC_FP32),
                                   (2048, 3, 1024, "ladder", chym.PREC_BF16X2)])
def test_batch_with_other_kernels_takes_no_longer_than_its_parts(other):
    """A large-N context beside one that runs in FP64, plain FP32 or over sparse rows."""
    torch = pytest.importorskip("torch")
    steps, sched = 400, chym.Schedule(1, 1000, 2000)
    N, D, R, kind, prec = other
    ctxs = [chym.Context(inputs.mobius_ladder(N) if kind == "ladder" else inputs.sk_pm1(N, 3), D),
            chym.Context(inputs.sk_pm1(1000, 3), 4)]
    prm = [chym.Params(eps=0.02, prec=prec), chym.Params(eps=0.008, prec=chym.PREC_BF16X2)]
    for c, p, runs in zip(ctxs, prm, (R, 2048)):
        c.run(p, np.array([0.8]), inputs.run_seeds(4, runs), 0, sched)

    def ms(of):
        b, t = chym.Batch([ctxs[i] for i in of]), []
        for _ in range(5):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            b.run([prm[i] for i in of], [sched] * len(of), steps, torch.cuda.current_stream().cuda_stream)
            t1.record()
            torch.cuda.synchronize()
            t.append(t0.elapsed_time(t1))
        b.status()
        b.close()
        return sorted(t)[2]

    both, small, large = ms([0, 1]), ms([0]), ms([1])
    assert both < 1.15 * (large + small), (both, large, small)
    for c in ctxs:
        c.close()

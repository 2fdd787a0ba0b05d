"""The batch tuner: its search starts from the shapes that an untuned batch takes, and a cached
tuning is taken only from the version of the cost model it was measured with."""
import json

import numpy as np
import pytest

from paper_2308_02329_gb300 import chym, inputs

pytestmark = pytest.mark.gpu


def _batch(specs, steps):
    """Contexts (N, D, R) with a state and a batch over them; params and schedules."""
    ctxs, prm = [], []
    sched = chym.Schedule(1, 10 * steps, 20 * steps)
    for i, (N, D, R) in enumerate(specs):
        ctx = chym.Context(inputs.gaussian(N, 3 + i), D, chym.J_REAL)
        prm.append(chym.Params(eps=0.25, prec=chym.PREC_BF16X2))
        ctx.run(prm[i], np.array([0.8]), inputs.run_seeds(i, R), 0, sched)
        ctxs.append(ctx)
    return ctxs, chym.Batch(ctxs), prm, [sched] * len(ctxs)


@pytest.mark.parametrize("specs", [
    [(250, 3, 1024)],                # few tiles: the default is narrower than any shape to choose
    [(250, 3, 256), (300, 3, 100)],
    [(100, 3, 2048)], [(60, 2, 500), (100, 2, 300)]])   # chunks of four and of eight runs
def test_tuned_is_not_slower_than_untuned(specs):
    torch = pytest.importorskip("torch")
    steps = 300
    ctxs, batch, prm, sched = _batch(specs, steps)

    def ms():
        best = np.inf
        for _ in range(6):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            batch.run(prm, sched, steps, torch.cuda.current_stream().cuda_stream)
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1))
        batch.status()
        return best

    untuned = ms()
    batch.tune(prm, sched, probe_steps=100)
    assert ms() < 1.1 * untuned
    batch.close()
    for c in ctxs:
        c.close()


def test_cached_tuning_of_another_cost_model_is_not_taken(tmp_path):
    """An entry without the version (written before there was one) is measured anew and kept."""
    ctxs, batch, prm, sched = _batch([(100, 3, 64), (200, 2, 40)], 20)
    path = tmp_path / "tuning.json"
    old = {"chunk": [123.0] * 8, "k2": 456.0, "shapes": {"rt": [32] * 8, "stages": [2] * 8, "ch": [0] * 8}}
    path.write_text(json.dumps({batch.signature("gpu"): old}))
    t = batch.tune(prm, sched, probe_steps=4, cache_path=str(path), device_key="gpu")
    assert t["chunk"] != old["chunk"] and t["k2"] != old["k2"]
    cache = json.loads(path.read_text())
    assert cache.pop(batch.signature("gpu")) == old and len(cache) == 1
    other = chym.Batch(ctxs)
    assert other.tune(prm, sched, probe_steps=4, cache_path=str(path), device_key="gpu")["chunk"] == t["chunk"]
    other.close()
    batch.close()
    for c in ctxs:
        c.close()

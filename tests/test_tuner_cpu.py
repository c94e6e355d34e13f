"""The autotuner on 2D grids whose gradients take several steps per launch: the
tiling has no part in them, so what it picks must come from the one-step
kernels that it governs (no GPU; the timing is faked)."""
import json

import pytest

torch = pytest.importorskip("torch")

from paper_2509_15744_gb300 import tune


class _Model:
    def __init__(self, shape, storage="f32", kahan=True):
        self.shape, self.order, self.physics, self.storage, self.kahan = shape, 4, "velocity", storage, kahan
        self.param = torch.zeros(1)
        self.tiling, self.timed = None, []

    def pitched_shape(self):
        return (self.shape[0], -(-self.shape[1] // 128) * 128)

    def set_tiling(self, *t):
        self.tiling = tuple(t)

    def set_schedule(self, order):
        pass

    def gradient(self, shots, **kw):
        self.timed.append("gradient")

    def step(self, cur, prev, acc=None, comp=None):
        assert all(tuple(t.shape) == self.pitched_shape() for t in cur + prev + [acc] + [comp] * self.kahan)
        assert cur[0] is not prev[0] and (comp is not None) == self.kahan
        self.timed.append("step")


def _tune(monkeypatch, tmp_path, model):
    """Tuned tiling where the one-step kernel is fastest at 2 rows per warp and
    a gradient call, which the tiling does not change, looks fastest at 128."""
    ms = {("step", 2): 1.0, ("gradient", 128): 1.0}
    monkeypatch.setattr(tune, "CACHE", str(tmp_path / "cache.json"))
    monkeypatch.setattr(tune.torch.cuda, "synchronize", lambda *a: None)
    monkeypatch.setattr(tune.W, "timing_enable", lambda on: None)
    monkeypatch.setattr(tune.W, "timing_read", lambda: (ms.get((model.timed[-1], model.tiling[0]), 2.0), 1, 0.0))
    return tune.tune(model, [tune.W.Shot(0, torch.zeros(31), torch.zeros(4, dtype=torch.int64))])


@pytest.mark.parametrize("kahan", [False, True])
def test_grids_of_several_steps_per_launch_are_tuned_by_single_steps(monkeypatch, tmp_path, kahan):
    m = _Model((300, 400), kahan=kahan)
    # what an earlier tuner kept for this grid was picked by noise
    old = json.dumps([2, [300, 400], 4, "velocity", "f32", kahan, 1])
    (tmp_path / "cache.json").write_text(json.dumps({old: [128, 8, 3, 0, 1]}))
    assert _tune(monkeypatch, tmp_path, m)[0] == 2 and m.tiling[0] == 2
    assert set(m.timed) == {"step"}
    m.timed.clear()
    assert _tune(monkeypatch, tmp_path, m)[0] == 2 and not m.timed   # kept


@pytest.mark.parametrize("shape,storage", [((300, 100), "f32"), ((300, 400), "bf16"), ((15, 400), "f32")])
def test_grids_of_one_step_per_launch_are_tuned_by_gradients(monkeypatch, tmp_path, shape, storage):
    m = _Model(shape, storage)
    assert _tune(monkeypatch, tmp_path, m)[0] == (128 if shape[0] >= 128 else m.tiling[0])
    assert set(m.timed) == {"gradient"}

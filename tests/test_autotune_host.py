"""The autotuner's choices (no GPU: timings are given)."""
import pytest

torch = pytest.importorskip("torch")

from paper_1504_01883_gb300 import autotune, binding as B  # noqa: E402


class Knobs:
    def __init__(self):
        self.value = {}

    def set_tuning(self, key, value):
        self.value[key] = value

    def layout(self):
        return self.value[B.TUNE_LBP_SHAPE], self.value[B.TUNE_LBP_CTAS_PER_SM]


def _tune(monkeypatch, times, cache=None):
    ctx = Knobs()
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "gpu")
    monkeypatch.setattr(autotune, "_load_cache", lambda: dict(cache or {}))
    monkeypatch.setattr(autotune, "_store_cache", lambda c: None)
    monkeypatch.setattr(autotune, "_time", lambda fn, stream, reps=3: times.get(ctx.layout(), 1.0))
    return autotune.tune(ctx, "k", None, None, 1, 1, None, tensor_core=False)[0], ctx


@pytest.mark.parametrize("times,want", [({}, (0, 0)), ({(2, 2): 0.99}, (0, 0)), ({(1, 1): 0.5}, (1, 1)),
                                        ({(1, 2): 0.9, (3, 1): 0.89}, (3, 1))])
def test_the_librarys_own_layout_stays_unless_another_is_clearly_faster(monkeypatch, times, want):
    t, ctx = _tune(monkeypatch, times)
    assert (t.lbp_shape, t.lbp_ctas_per_sm) == want == ctx.layout()


def test_choices_cached_for_earlier_kernels_are_not_used(monkeypatch):
    old = {f"gpu|{v}|k": {"tuning": {"lbp_ctas_per_sm": 1, "lbp_shape": 1}} for v in range(5)}
    t, _ = _tune(monkeypatch, {}, old)
    assert (t.lbp_shape, t.lbp_ctas_per_sm) == (0, 0)

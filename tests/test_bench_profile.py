"""The bench's per-step kernel times come from steps after a warm-up."""
import bench


class FakeLibrary:
    """Counts steps; records one launch a step while profiling is on, the first
    step ever twenty times as slow."""

    def __init__(self):
        self.on, self.steps, self.record = False, 0, {}

    def step(self):
        self.steps += 1
        if self.on:
            c, t = self.record.get("k", (0, 0.0))
            self.record["k"] = (c + 2, t + (20.0 if self.steps == 1 else 1.0))

    def wo_profile_enable(self, on):
        self.on = on

    def wo_profile_read(self):
        r, self.record = self.record, {}
        return r


def test_step_profile_is_per_step_and_warm(monkeypatch):
    import torch
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a: None)
    lib = FakeLibrary()
    assert bench.step_profile(lib, lib.step, warmup=3, n=5) == {"k": (2, 1.0)}
    assert lib.steps == 8 and not lib.on


def test_the_tuning_leg_profiles_warm_steps():
    """The leg has no profile of its own beside step_profile."""
    import inspect
    src = inspect.getsource(bench.autotune_leg)
    assert "step_profile(" in src and "wo_profile_enable" not in src

"""Combinations that differ in choices a context names inert share one timing,
and such a choice keeps its default."""
from paper_2408_14140_gb300 import api, autotune


class Inert:
    INERT_CHOICES = api.Context.INERT_CHOICES

    def __init__(self):
        self.stages = set()

    def set_pass_kernels(self, which):
        pass

    def set_volume_split(self, n):
        pass

    def set_gather(self, ctas, stage):
        self.stages.add(stage)


def test_inert_choices_are_not_timed(monkeypatch):
    ctx, timed = Inert(), []
    monkeypatch.setattr(autotune, "time_step", lambda step, **kw: timed.append(1) or 1.0 / len(timed))
    out = autotune.tune([ctx], step=lambda: None)
    assert ctx.stages == {0} and out["choice"]["gather_stage"] == 0
    assert set(out["choice"]) == set(autotune.SPACE)
    effects = {tuple(sorted((k, v) for k, v in c.items() if k != "gather_stage")) for c, _ in out["table"]}
    assert len(effects) == len(timed) < len(out["table"])

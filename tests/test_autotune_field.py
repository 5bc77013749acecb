"""The complex64 field has one path: the autotuner prepares and times it once."""

from test_autotune import FakeCav, FakeTimer

from paper_2008_01966_gb300 import autotune


def test_one_field_path_is_timed():
    cav = FakeCav(256)
    fields = []
    cav.field = fields.append
    timer = FakeTimer(cav, {"b": {0: 0.0}, "c": {0: 0.0}, "g": {16: 3.0, 8: 2.0, 4: 1.0}})
    out = autotune.tune(cav, 1.0, [(16, 1.0)], [0.1], [0.0], [0.0], reps=1, timer=timer)
    assert len(fields) == 1 and len(out["ms"]["field_fused"]) == 1
    assert cav.prepared == 2          # the option's prepare, and the one the other options start from
    assert out["choice"]["field_fused"] == 1 and out["choice"]["group_width"] == 8

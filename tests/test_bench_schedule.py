"""The sweep schedule that bench.py names is the one that it asks for."""
import bench


def test_global_is_asked_for_by_name():
    """A default plan may take the range schedule: the level-ordered kernel has to be asked for."""
    g, p = bench.Schedule("global", 16, "cpu", None), bench.Schedule.__new__(bench.Schedule)
    p.kind = "part"
    assert g.plan_args() == {"schedule": "global"} and p.plan_args() == {}
    assert g.kernel().startswith("k_sweep<") and p.kernel().startswith("k_sweep_part<")


def test_tuned_schedules_are_named_as_reported():
    tuned = lambda *kinds: [{"schedule": k} for k in kinds]  # noqa: E731
    assert bench.tuned_schedule(tuned("range", "range"), 256).startswith("ranges (")
    assert bench.tuned_schedule(tuned("part", "part"), 256).startswith("x-pencil partitioned, 256 parts (")
    assert bench.tuned_schedule(tuned("global", "range"), 256).startswith("L global, U ranges (")

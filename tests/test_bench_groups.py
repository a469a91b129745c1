"""bench.py's traffic figure of grouped steps, without a GPU: given only for what
its capture measured, periods of about as many steps of a full buffer and no
densities in the groups, from the kernel source as it is."""
import bench

DELTA = {"particle_steps": 10_000_000, "eventful": 200_000, "spawned": 30, "injected": 0}


def test_group_traffic_is_given_for_what_was_captured(monkeypatch):
    monkeypatch.setattr(bench, "NCU_GROUP", {"bytes": 0.5, "steps": 50, "src_sha": bench.kernel_sha("pic_group.cu")})
    kt = {"step": (26, 8.0), "step_moments": (2, 0.5), "step_events": (26, 0.5)}
    assert bench.group_traffic(DELTA, kt, 100) == 0.5 * 10_000_000 / 100
    assert bench.group_traffic(dict(DELTA, spawned=100_000), kt, 100) is None
    assert bench.group_traffic(dict(DELTA, injected=100_000), kt, 100) is None
    # densities inside the groups: every pass counts as one with densities
    assert bench.group_traffic(DELTA, dict(kt, step=(0, 0.0), step_moments=(25, 8.0)), 100) is None
    # windows of 10 steps, or none in the time
    assert bench.group_traffic(DELTA, dict(kt, step_moments=(10, 0.5)), 100) is None
    assert bench.group_traffic(DELTA, dict(kt, step_moments=(0, 0.0)), 100) is None
    monkeypatch.setitem(bench.NCU_GROUP, "src_sha", "0" * 16)
    assert bench.group_traffic(DELTA, kt, 100) is None

"""When executions and batches take the channel-group kernel, and when its table
is built: host code on stand-ins for 152 SMs, no GPU."""
import numpy as np
import pytest

from tests import hostrt
from tests.hostrt import DIRECT, GROUPED, TABLE


@pytest.fixture()
def host():
    h = hostrt.Host()
    yield h
    h.lib.fake_capturing(0)
    h.reset()


def _narrow(host, nchan, ndm, step=1.0):
    return host.plan(nchan, 1500.0, -64.0 / nchan, 64e-6, step * np.arange(ndm))


def _lband(host, nchan, ndm):
    return host.plan(nchan, 1500.0, -300.0 / nchan, 64e-6, np.arange(ndm))


def _kinds(host, call, *args):
    host.reset()
    assert call(*args) == 0
    return [r.kind for r in host.records()]


def test_a_long_execution_builds_its_table_first(host):
    plan = _narrow(host, 1024, 1024)
    assert _kinds(host, host.execute, plan, "u8", 65536) == [TABLE, GROUPED]
    assert _kinds(host, host.execute, plan, "u8", 65536) == [GROUPED]


def test_a_short_execution_builds_its_table_behind_the_direct_kernel(host):
    """It gains some 100 us, less than the table costs it."""
    plan = _narrow(host, 1024, 128)
    assert _kinds(host, host.execute, plan, "u8", 61440) == [DIRECT, TABLE]
    assert _kinds(host, host.execute, plan, "u8", 61440) == [GROUPED]


def test_a_table_under_way_is_not_waited_for(host):
    plan = _narrow(host, 1024, 128)
    _kinds(host, host.execute, plan, "u8", 61440)
    host.lib.fake_tables(1, 0)
    assert host.execute(plan, "u8", 61440) == 0
    host.lib.fake_tables(1, 1)
    assert host.execute(plan, "u8", 61440) == 0
    assert [r.kind for r in host.records()] == [DIRECT, TABLE, DIRECT, GROUPED]


def test_a_capture_waits_for_the_table(host):
    """The graph keeps the kernel that it captures."""
    plan = _narrow(host, 1024, 128)
    host.lib.fake_tables(1, 0)
    host.lib.fake_capturing(1)
    assert _kinds(host, host.execute, plan, "u8", 61440) == [TABLE, GROUPED]


def test_unusable_tables_leave_the_direct_kernel(host):
    plan = _narrow(host, 1024, 1024)
    host.reset()
    host.lib.fake_tables(0, 1)
    for _ in range(3):
        assert host.execute(plan, "u8", 65536) == 0
    kinds = [r.kind for r in host.records()]
    assert GROUPED not in kinds and kinds.count(DIRECT) == 3 and kinds.count(TABLE) <= 2


def test_no_memory_for_the_table_leaves_the_direct_kernel(host):
    plan = _narrow(host, 1024, 1024)
    assert host.execute(plan, "u8", 64) == 0  # the plan's own tables
    for _ in range(2):
        host.lib.fake_fail_malloc(1)
        assert host.execute(plan, "u8", 65536) == 0
    assert not [r for r in host.records(DIRECT, GROUPED) if r.null_pointers]


def test_destroying_a_plan_gives_its_table_back(host):
    before = host.lib.fake_allocations()
    for done in (1, 0):
        plan = _narrow(host, 1024, 128)
        host.reset()
        host.lib.fake_tables(1, done)
        assert host.execute(plan, "u8", 61440) == 0
        assert host.records(TABLE)
        host.lib.dd_plan_destroy(plan)
    assert host.lib.fake_allocations() == before


def test_a_batch_of_one_round_stays_direct(host):
    """3 beams of 100 DMs: 144 direct tiles are one round, 96 grouped ones take
    longer each (measured 306 and 383 us)."""
    batch = host.batch([_lband(host, 1024, 100) for _ in range(3)], "u8", [16384] * 3)
    for _ in range(2):
        assert GROUPED not in _kinds(host, host.batch_execute, batch)


def test_a_short_batch_builds_its_tables_behind_its_first_execution(host):
    batch = host.batch([_lband(host, 1024, 24) for _ in range(8)], "u8", [16384] * 8)
    assert _kinds(host, host.batch_execute, batch) == [DIRECT] + 8 * [TABLE]
    second = _kinds(host, host.batch_execute, batch)
    assert TABLE not in second and GROUPED in second
    captured = [r.captured for r in host.records(GROUPED)]
    assert captured == [0, 1]  # eager, then into the graph


def test_a_batch_does_not_wait_for_tables_under_way(host):
    batch = host.batch([_lband(host, 1024, 24) for _ in range(8)], "u8", [16384] * 8)
    host.reset()
    host.lib.fake_tables(1, 0)
    for _ in range(3):
        assert host.batch_execute(batch) == 0
    assert [r.kind for r in host.records(DIRECT, GROUPED)] == 3 * [DIRECT]
    assert len(host.records(TABLE)) == 8
    host.lib.fake_tables(1, 1)
    assert GROUPED in _kinds(host, host.batch_execute, batch)


def test_a_long_batch_builds_its_tables_together(host):
    """All tables are under way before the batch waits for one."""
    batch = host.batch([_narrow(host, 1024, 1024) for _ in range(4)], "u8", [65536] * 4)
    kinds = _kinds(host, host.batch_execute, batch)
    assert kinds[:5] == 4 * [TABLE] + [GROUPED]


def test_batch_with_unusable_tables(host):
    batch = host.batch([_narrow(host, 1024, 1024) for _ in range(2)], "u8", [65536] * 2)
    host.reset()
    host.lib.fake_tables(0, 1)
    for _ in range(3):
        assert host.batch_execute(batch) == 0
    launches = host.records(DIRECT, GROUPED)
    assert {r.kind for r in launches} == {DIRECT} and not any(r.null_pointers for r in launches)


@pytest.mark.parametrize("kind", ["u8", "f16", "f32"])
def test_a_replayed_batch_counts_the_kernels_that_its_graph_holds(host, kind):
    """dd_launch_count: the same for the eager execution as for the graph's."""
    plans = [_narrow(host, 1024, 1024), _lband(host, 64, 40), _lband(host, 64, 40)]
    batch = host.batch(plans, kind, [65536, 8192, 8192])
    host.lib.dd_launch_count.restype = hostrt.ctypes.c_int64
    counts = []
    for _ in range(3):
        before = host.lib.dd_launch_count()
        assert host.batch_execute(batch) == 0
        counts.append(host.lib.dd_launch_count() - before)
    assert counts == 3 * [2 if kind == "u8" else 1]

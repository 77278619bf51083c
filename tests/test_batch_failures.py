"""A batch whose allocations fail: the call returns the error, and a later call
goes on with everything it needs.  Host code on stand-ins, no GPU."""
import numpy as np
import pytest

from tests import hostrt

NOMEM = -3


@pytest.fixture()
def host():
    h = hostrt.Host()
    yield h
    h.reset()


@pytest.mark.parametrize("kind", ["u8", "f32"])
@pytest.mark.parametrize("nth", range(1, 16))
def test_a_failed_allocation_leaves_no_null_pointers(host, kind, nth):
    plans = [host.plan(64, 1500.0, -300.0 / 64, 64e-6, np.arange(40)),
             host.plan(1024, 1500.0, -64.0 / 1024, 64e-6, np.arange(200))]
    batch = host.batch(plans, kind, [8192, 65536])
    host.reset()
    host.lib.fake_fail_malloc(nth)
    first = host.batch_execute(batch)
    assert first in (0, NOMEM)
    if first == NOMEM:
        assert not host.records(hostrt.DIRECT, hostrt.GROUPED)
    for _ in range(2):
        assert host.batch_execute(batch) == 0
    launches = host.records(hostrt.DIRECT, hostrt.GROUPED)
    assert launches and not any(r.null_pointers for r in launches)
    host.lib.dd_batch_destroy(batch)

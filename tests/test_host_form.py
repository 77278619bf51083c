"""dd_execute_host on stand-ins: the order of its work, without a GPU."""
import numpy as np

from tests import hostrt
from tests.hostrt import GROUPED, H2D, TABLE


def test_the_table_is_built_behind_the_first_input_copy():
    host = hostrt.Host()
    plan = host.plan(1024, 1500.0, -64.0 / 1024, 64e-6, np.arange(1024))
    host.reset()
    assert host.execute(plan, "u8", 131072, host=True) == 0
    kinds = [r.kind for r in host.records()]
    assert kinds[:3] == [H2D, TABLE, GROUPED] and kinds.count(TABLE) == 1

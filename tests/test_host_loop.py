"""When the host loop (host_loop = 1) stops launching iterations (no GPU needed):
a timeout ends it whatever the stop word holds, since launches after a timeout
return at once and would never set it."""
import pytest

import device_probe
from paper_2510_08536_gb300 import repart


@pytest.mark.parametrize("stop,status,runs", [
    (0, -1, 1),
    (1, -1, 0),
    (1, repart.RP_DEVICE_TIMEOUT, 0),
    (0, repart.RP_DEVICE_TIMEOUT, 0),
    (1, repart.RP_BREAKDOWN, 0),
])
def test_host_loop_decision(stop, status, runs):
    assert device_probe.load().probe_inner_runs(stop, status) == runs

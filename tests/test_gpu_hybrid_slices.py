"""Sliced hybrid walks: every packet is emitted once and ends once, however the
walk is cut."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1709_10187_gb300 import build as B  # noqa: E402
from paper_1709_10187_gb300 import rddmc as R  # noqa: E402
from paper_1709_10187_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
COUNTS = ("emitted", "escaped", "aborted", "steps", "event_draws", "mc_events", "conversions", "clamps")


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def _same(a, b):
    for k in COUNTS:
        assert a[k] == b[k], (k, a[k], b[k])
    for k in ("hist", "faces", "sb"):
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("w", [
    W.Workload("thin_slab", 1, (8, 1, 1), 16, -8.0, 8.0, 4.0, 1.0e4, 3000, 0x5EED0D01),
    W.Workload("mixed_slab", 1, (9, 1, 1), 12, -6.0, 6.0, 30.0, 1.0e4, 3000, 0x5EED0D02),
    W.Workload("mixed_sphere", 3, (7, 7, 7), 12, -6.0, 6.0, 20.0, 1.0e4, 3000, 0x5EED0D03, sphere=True, vmax_kms=30.0),
], ids=lambda w: w.name)
def test_packets_that_end_in_their_source_excursion_are_emitted_once(w):
    # a thin source state starts as MC, and the packet may escape before its first
    # transition; tau_ddmc between the cells' depths mixes thin and thick states
    p = R.Problem(w, mode=R.MODE_HYBRID)
    n = w.packets
    one = p.run(n, w.seed)
    assert one["emitted"] == one["escaped"] == n
    p.reset()
    p.launch(n, w.seed, steps_per_launch=8)
    first = p.packet_states(n, 0, n)
    done = p.read()["escaped"]
    assert done > 0 and (first["status"] == 2).sum() == done
    for _ in range(3):
        p.launch(n, w.seed, steps_per_launch=8, resume=1)
    p.launch(n, w.seed, steps_per_launch=1 << 40, resume=1)
    _same(p.read(), one)
    p.close()

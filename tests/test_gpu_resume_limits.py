"""Watchdog limits that change between the launches of a run: a packet resumed
past the limit is aborted before it takes another transition."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1709_10187_gb300 import build as B  # noqa: E402
from paper_1709_10187_gb300 import rddmc as R  # noqa: E402
from paper_1709_10187_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


@pytest.mark.parametrize("w", [W.SMALL, W.SPHERE8_V], ids=lambda w: w.name)
def test_time_step_with_a_lower_limit_aborts_at_once(w):
    p, n = R.Problem(w), 3000
    state = torch.empty(R.time_state_bytes(n), dtype=torch.uint8, device="cuda")
    S = w.ncell * p.J
    bins, path = (torch.zeros((3, S), dtype=torch.int64, device="cuda") for _ in range(2))
    counts = torch.zeros((3, 5), dtype=torch.int64, device="cuda")
    p.reset()

    def step(k, limit):
        R.time_step_launch(p.grid, p.table.data_ptr(),
                           R.TimeStep(w.seed, n, limit, 0.05 * k, 0.05 * (k + 1), int(k == 0), 0, 0, 0, 0),
                           state.data_ptr(), state.numel(), p.tally.data_ptr(), p.tally.numel() * 8,
                           bins[k].data_ptr(), path[k].data_ptr(), counts[k].data_ptr(), p.stream())

    step(0, 0)
    before = p.read()
    s = R.read_packet_states(p.grid, state.data_ptr(), n, 0, n)
    flying = s["status"] == 1
    assert flying.sum() > n // 2 and s["steps"][flying].max() > s["steps"][flying].min() + 8
    limit = int(np.median(s["steps"][flying]))
    over = int((s["steps"][flying] >= limit).sum())
    step(1, limit)
    esc, dwells, moves, alive, _ = counts[1].cpu().numpy()
    t = p.read()
    # those past the limit are gone without a dwell, the others walk up to it
    assert over <= t["aborted"] <= flying.sum()
    assert t["aborted"] + esc + alive == flying.sum()
    assert dwells == moves + alive
    s1 = R.read_packet_states(p.grid, state.data_ptr(), n, 0, n)
    assert np.all(s1["status"][flying & (s["steps"] >= limit)] == 2)
    assert np.all(s1["steps"][s1["status"] == 1] < limit)
    assert moves <= (limit - s["steps"][flying & (s["steps"] < limit)]).sum()
    assert t["steps"] - before["steps"] == moves
    # of those left only packets that have not moved yet can, once
    step(2, 1)
    left = p.read()
    esc, dwells, moves, stay, _ = counts[2].cpu().numpy()
    unmoved = int((s1["steps"][s1["status"] == 1] == 0).sum())
    assert moves <= unmoved and stay <= unmoved and dwells == moves + stay
    assert left["aborted"] - t["aborted"] + esc + stay == alive
    assert int(bins[2].sum()) == stay and left["steps"] - t["steps"] == moves
    p.close()

"""Limits of the launches of a run.  Watchdog limits that change between them: a
packet resumed past the limit is aborted before it takes another transition.
Wall-time slices end on time whatever number of CTAs is asked for."""
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


PATHS = ["pairs", "heads", "hybrid", "hybrid thick", "weights", "cube", "rows", "thick moving", "proposal"]


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("limit", [1, 63, 64, 97])
def test_walk_with_a_lower_limit_aborts_at_once(path, limit):
    # every way of reading transitions: pairs, heads (a table past the pairs' row
    # count, a hybrid slab, the weight method), rows, and parking for a proposal
    cube = W.Workload("limit_cube", 3, (8, 8, 8), 16, -9.0, 9.0, 2.0e5, 1.0e4, 1, 0x5EED0C01)
    kw = {}
    if path == "pairs":
        w = W.C1
    elif path == "heads":
        w, kw = W.Workload("limit_dense", 1, (2050, 1, 1), 512, -60.0, 60.0, 1.0e8, 1.0e4, 1, 1), dict(
            layout=R.LAYOUT_DENSE)
    elif path.startswith("hybrid"):
        w, kw = W.C1.with_(tau0=2.0e6 if path == "hybrid thick" else 1.0e5), dict(mode=R.MODE_HYBRID)
    elif path == "weights":
        w, kw = W.C1, dict(dust_abs=1e-3, dust_weights=True)
    else:
        w = {"rows": cube.with_(tau0=1.0e3, vmax_kms=30.0), "thick moving": cube.with_(vmax_kms=30.0)}.get(path, cube)
    n, first = 3000, 128
    p = R.Problem(w, **kw)
    prop, keep = None, []
    if path == "proposal":  # one whole brick whose packets are never served (no eligible brick)
        t = lambda *a, **k: keep.append(torch.tensor(*a, device="cuda", **k)) or keep[-1].data_ptr()  # noqa: E731
        prop = R.Proposal()
        prop.brick, prop.margin, prop.n_bricks = 8, 1, 1
        prop.d_brick_lk, prop.d_lp, prop.d_xc = t([-1e30]), t([0.0] * 16), t([0.0] * 16)
        prop.d_queue_count, prop.d_queue_pid = t([0], dtype=torch.int64), t([0] * n, dtype=torch.int64)
    p.reset()
    p.launch(n, 5, steps_per_launch=first, proposal=prop)
    a, s = p.read(), p.packet_states(n, 0, n)
    flying = s["status"] == 1
    assert flying.sum() > 100 and np.all(s["steps"][flying] == first)
    p.launch(n, 5, steps_per_launch=first, resume=1, max_steps=limit, proposal=prop)
    b = p.read()
    assert b["aborted"] - a["aborted"] == flying.sum()
    for k in ("emitted", "escaped", "steps", "mc_events", "event_draws", "absorbed"):
        assert a[k] == b[k], k
    assert np.all(p.packet_states(n, 0, n)["status"] == 2)
    p.close()


@pytest.mark.parametrize("ctas,threads", [(0, 0), (4, 256), (12, 256), (24, 128)])
def test_wall_time_slices_are_not_repeated_by_waiting_ctas(ctas, threads):
    p, n, ms = R.Problem(W.C1), 500_000, 20.0
    p.reset()
    p.launch(n, 5, steps_per_launch=64)
    took = []
    for _ in range(3):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        p.launch(n, 5, resume=1, time_slice_us=int(1e3 * ms), ctas_per_sm=ctas, threads_per_cta=threads)
        b.record()
        torch.cuda.synchronize()
        took.append(a.elapsed_time(b))
    assert ms <= min(took) < 1.6 * ms, took
    assert (p.packet_states(n, 0, n)["status"] == 1).sum() > n // 2
    p.close()

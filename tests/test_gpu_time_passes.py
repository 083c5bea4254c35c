"""Passes of the time-dependent walk: a lane takes the rest of its block of four
transition words with the dwell words that go with them, whatever the offsets
of the two (t mod 4, and the steps survived mod 4), the watchdog's limit and the
points at which warps regroup or refill."""
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


@pytest.mark.parametrize("max_steps", [0, 1, 2, 3, 4, 5, 6, 7, 30])
@pytest.mark.parametrize("w", [W.SMALL, W.SPHERE8_V], ids=lambda w: w.name)
def test_results_do_not_depend_on_chunks_or_regrouping(w, max_steps):
    p = R.Problem(w)
    n, te = 3000, [0.0, 0.02, 0.05, 0.1, 0.15, 0.2, 0.25, 0.4]  # steps survived 0 .. 6
    ref = p.time_run(n, w.seed, te, max_steps=max_steps, chunk=4, regroup=-1)
    if max_steps:
        assert ref["tallies"]["steps"] <= max_steps * n and ref["tallies"]["aborted"] > 0
    # a packet is alive at a step's end, or has left by then
    gone = np.cumsum(ref["esc"].astype(np.int64))
    alive = ref["alive"].astype(np.int64)
    assert np.all(alive + gone <= n) and np.all(np.diff(alive) <= 0)
    assert alive[-1] + ref["tallies"]["escaped"] + ref["tallies"]["aborted"] == n
    # every dwell ends in a transition or stops a packet at the step's end
    assert np.array_equal(ref["dwells"], ref["transitions"] + ref["alive"])
    for kw in (dict(chunk=8, regroup=32), dict(chunk=256, regroup=1), dict(threads_per_cta=32, ctas_per_sm=1), dict()):
        r = p.time_run(n, w.seed, te, max_steps=max_steps, **kw)
        for k in ("bins", "path_ticks", "esc", "dwells", "transitions", "alive"):
            assert np.array_equal(r[k], ref[k]), (kw, k)
        for k in ("emitted", "escaped", "aborted", "steps", "clamps", "event_draws"):
            assert r["tallies"][k] == ref["tallies"][k], (kw, k)
        assert np.array_equal(r["tallies"]["hist"], ref["tallies"]["hist"])
    p.close()

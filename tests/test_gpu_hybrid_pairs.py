"""Hybrid slabs on either side of the cell depth (4e4) from which they read pairs:
excursions that change cell, class and state in the middle of a group of four."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import analytic as A  # noqa: E402
from oracle import coracle as C  # noqa: E402
from paper_1709_10187_gb300 import build as B  # noqa: E402
from paper_1709_10187_gb300 import rddmc as R  # noqa: E402
from paper_1709_10187_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
COUNTS = ("emitted", "escaped", "aborted", "steps", "event_draws", "mc_events", "conversions")


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def _same(a, b):
    for k in COUNTS:
        assert a[k] == b[k], (k, a[k], b[k])
    assert np.array_equal(a["hist"], b["hist"]) and np.array_equal(a["faces"], b["faces"])


def _slab(depth, v=0.0, **kw):
    return W.Workload("hybrid_pairs", 1, (6, 1, 1), 24, -30.0, 30.0, 3.0 * depth, 1.0e4, 3000, 0x5EED1001,
                      vmax_kms=v).with_(**kw)


@pytest.mark.parametrize("depth", [3.0e4, 5.0e4, 3.0e5])
def test_all_thick_hybrid_is_the_ddmc_walk(depth):
    w = _slab(depth)
    a = R.Problem(w).run(w.packets, w.seed)
    b = R.Problem(w, mode=R.MODE_HYBRID, tau_ddmc=1e-30).run(w.packets, w.seed)
    assert a["escaped"] == w.packets and b["mc_events"] == 0
    _same(a, b)


@pytest.mark.parametrize("grouped", [False, True])
def test_pairs_and_heads_walk_alike(grouped):
    # the dense table is past 2^20 rows and reads heads, the deduplicated one pairs;
    # bins past three Doppler widths are thin, and packets make excursions there
    w = W.Workload("hybrid_dense", 1, (2050, 1, 1), 512, -60.0, 60.0, 4.5e7, 1.0e4, 3000, 0x5EED1002)
    out = []
    for layout in (R.LAYOUT_DENSE, R.LAYOUT_DEDUP):
        p = R.Problem(w, mode=R.MODE_HYBRID, layout=layout)
        redist = p.redistribution(1) if grouped else None
        assert (p.sizes.n_class * p.J > 1 << 20) == (layout == R.LAYOUT_DENSE)
        p.reset()
        for k in range(3):
            p.launch(w.packets, w.seed, steps_per_launch=20_000, resume=int(k > 0), max_steps=59_998, redist=redist)
        out.append((p.read(), p.packet_states(w.packets, 0, w.packets)))
        p.close()
    (a, sa), (b, sb) = out
    assert a["mc_events"] > 1000 and a["conversions"] > 0
    _same(a, b)
    for k in sa:
        assert np.array_equal(sa[k], sb[k]), k


@pytest.mark.parametrize("depth,v", [(3.0e4, 0.0), (5.0e4, 0.0), (5.0e4, 30.0), (3.0e5, 0.0)])
def test_slices_equal_one_launch_and_the_spectrum_matches_the_oracle(depth, v):
    w = _slab(depth, v)
    p = R.Problem(w, mode=R.MODE_HYBRID)
    one = p.run(w.packets, w.seed)
    assert one["escaped"] == w.packets and one["mc_events"] > 0
    p.reset()
    for k in range(30):
        p.launch(w.packets, w.seed, steps_per_launch=12, resume=int(k > 0))
    p.launch(w.packets, w.seed, steps_per_launch=1 << 40, resume=1)
    _same(p.read(), one)
    p.close()
    n = w.packets
    og = C.Grid(w, hybrid=True)
    orc = C.walk(og, og.table(), w.seed + 11, 0, n)
    zmax, frac = A.compare_two_samples(one["hist"], n, orc["hist"], n)
    assert zmax < 5.0 and frac <= 0.05, (zmax, frac)
    for k in ("mc_events", "conversions", "steps"):
        g, o = one[k] / n, orc[k] / n
        assert abs(g - o) <= 0.1 * max(g, o) + 1.0, (k, g, o)

"""The walk's pair reads (two frequency moves per gather) against the oracle and
the fast-head walk: grids of a few bins, where every pair touches the grid's
ends, watchdog limits inside a group of four, slices, and the two sides of the
row count up to which a table carries pairs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import coracle as C  # noqa: E402
from paper_1709_10187_gb300 import build as B  # noqa: E402
from paper_1709_10187_gb300 import rddmc as R  # noqa: E402
from paper_1709_10187_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
COUNTS = ("emitted", "escaped", "aborted", "steps", "clamps", "event_draws")


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def _same(a, b, nf):
    for k in COUNTS:
        assert a[k] == b[k], k
    assert np.array_equal(a["hist"], b["hist"]) and np.array_equal(a["faces"][:nf], b["faces"][:nf])
    assert np.array_equal(a["sb"], b["sb"])


@pytest.mark.parametrize("max_steps", [0, 1, 7, 130, 259])
@pytest.mark.parametrize("ndim,J,v", [(1, 1, 0.0), (1, 2, 0.0), (1, 3, 0.0), (1, 5, 0.0), (3, 2, 0.0), (3, 3, 20.0),
                                      (3, 4, 20.0)])
def test_few_bins_and_odd_limits_match_the_oracle(ndim, J, v, max_steps):
    n = (5, 1, 1) if ndim == 1 else (6, 6, 6)
    w = W.Workload(f"pairs_{ndim}_{J}", ndim, n, J, -6.0, 6.0, 40.0, 1.0e4, 3000, 0x5EED0B01, sphere=ndim == 3,
                   vmax_kms=v)
    g = C.Grid(w)
    ot = g.table()
    p = R.Problem(w)
    thr, flags = p.rows()
    sel = np.ones(w.ncell * J, bool) if w.mask() is None else np.repeat(w.mask().astype(bool), J)
    ot["thr"][sel] = thr[sel]  # walk the device's own thresholds (equal to one count)
    gpu = p.run(w.packets, w.seed, max_steps=max_steps)
    orc = C.walk(g, ot, w.seed, 0, w.packets, max_steps=max_steps or 1 << 62)
    _same(gpu, orc, 2 * ndim)
    p.close()


@pytest.mark.parametrize("case", ["slab", "graded", "cube", "sphere", "layers"])
@pytest.mark.parametrize("max_steps", [0, 41])
def test_rows_in_groups_of_four_match_the_oracle(case, max_steps):
    # wing-heavy grids: most transitions are spatial moves on the rows, in cells
    # more and less than four moves inside their class, to the grid's ends, to
    # vacuum and between classes of different density
    n_rel, sphere = None, False
    if case in ("slab", "graded"):
        n, ndim = (24, 1, 1), 1
        if case == "graded":
            n_rel = np.linspace(0.5, 2.0, 24)
    else:
        n, ndim = ((11, 14, 9), 3) if case != "sphere" else ((13, 13, 13), 3)
        sphere = case == "sphere"
        if case == "layers":  # two media, six cells thick on average
            n_rel = np.where(np.arange(11 * 14 * 9) // 11 % 14 < 7, 1.0, 3.0)
    w = W.Workload(f"rows_{case}", ndim, n, 15, -45.0, 45.0, 2.0e3, 1.0e4, 4000, 0x5EED0B03, sphere=sphere)
    g = C.Grid(w, n_rel=n_rel)
    ot = g.table()
    p = R.Problem(w, n_rel=n_rel)
    thr, _ = p.rows()
    sel = np.ones(w.ncell * w.J, bool) if w.mask() is None else np.repeat(w.mask().astype(bool), w.J)
    ot["thr"][sel] = thr[sel]
    orc = C.walk(g, ot, w.seed, 0, w.packets, max_steps=max_steps or 1 << 62)
    _same(p.run(w.packets, w.seed, max_steps=max_steps), orc, 2 * ndim)
    # the batched walk takes the same path with its own lane's tables
    b = R.Batch([p, p], [w.packets, 7])
    b.launch(R.RunOpts(w.seed, 0, max_steps))
    _same(b.read(0), orc, 2 * ndim)
    p.close()


@pytest.mark.parametrize("chunk", [4, 12, 256])
def test_pairs_and_heads_walk_alike(chunk):
    # dense tables below and above 2^20 rows: pairs on one side, heads on the other
    for n, J in ((2047, 512), (2050, 512)):
        w = W.Workload(f"rows_{n}", 1, (n, 1, 1), J, -60.0, 60.0, 1.0e6, 1.0e4, 4000, 0x5EED0B02)
        assert (n * J > 1 << 20) == (n == 2050)
        dense, dedup = R.Problem(w, layout=R.LAYOUT_DENSE), R.Problem(w)
        out = []
        for p in (dense, dedup):
            p.reset()
            p.launch(w.packets, w.seed, max_steps=6002, steps_per_launch=3000, chunk=chunk)
            for _ in range(2):
                p.launch(w.packets, w.seed, max_steps=6002, steps_per_launch=3000, resume=1, chunk=chunk)
            out.append(p.read())
        assert out[0]["emitted"] == w.packets == out[0]["escaped"] + out[0]["aborted"]
        _same(out[0], out[1], 2)
        for p in (dense, dedup):
            p.close()


@pytest.mark.parametrize("case", ["slab", "cube", "sphere_moving"])
@pytest.mark.parametrize("dust", [0.0, 3.0])
def test_dusty_and_moving_rows_match_the_oracle(case, dust):
    # absorbed packets among the groups on the rows; rebins whose event words
    # come from a kept block, over slices that cut packets between them
    if case != "sphere_moving" and not dust:
        pytest.skip("covered above")
    ndim = 1 if case == "slab" else 3
    n = {"slab": (20, 1, 1), "cube": (9, 8, 10), "sphere_moving": (12, 12, 12)}[case]
    w = W.Workload(f"dust_{case}", ndim, n, 21, -42.0, 42.0, 1.0e3, 1.0e4, 4000, 0x5EED0B04,
                   sphere=case == "sphere_moving", vmax_kms=60.0 if case == "sphere_moving" else 0.0)
    g = C.Grid(w, dust_abs=dust)
    ot = g.table()
    p = R.Problem(w, dust_abs=dust)
    thr, _ = p.rows()
    sel = np.ones(w.ncell * w.J, bool) if w.mask() is None else np.repeat(w.mask().astype(bool), w.J)
    ot["thr"][sel] = thr[sel]
    orc = C.walk(g, ot, w.seed, 0, w.packets, max_steps=1 << 62)
    one = p.run(w.packets, w.seed)
    _same(one, orc, 2 * ndim)
    assert one["absorbed"] == orc["absorbed"] and (one["absorbed"] > 0) == (dust > 0.0)
    p.reset()
    p.launch(w.packets, w.seed, steps_per_launch=12)
    for _ in range(30):
        p.launch(w.packets, w.seed, steps_per_launch=12, resume=1)
    p.launch(w.packets, w.seed, steps_per_launch=1 << 40, resume=1)
    _same(p.read(), orc, 2 * ndim)
    p.close()


@pytest.mark.parametrize("moving", [False, True])
def test_small_launches_walk_every_packet_as_full_ones_do(moving):
    # the default launch shape on both sides of its lines: a lane per warp, one
    # and two warps per scheduler, a launch that just fills the chip
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = (W.Workload("few_sphere", 3, (6, 6, 6), 9, -9.0, 9.0, 60.0, 1.0e4, 1, 0x5EED0B05, sphere=True, vmax_kms=30.0)
         if moving else W.Workload("few_slab", 1, (8, 1, 1), 16, -8.0, 8.0, 200.0, 1.0e4, 1, 0x5EED0B05))
    p = R.Problem(w)
    for n in (1, 4 * sms, 4 * sms + 1, 128 * sms, 128 * sms + 1, 256 * sms, 256 * sms + 1, 768 * sms - 1, 768 * sms):
        got = p.run(n, w.seed)
        assert got["emitted"] == n == got["escaped"]
        _same(got, p.run(n, w.seed, threads_per_cta=256, ctas_per_sm=3), 2 * w.ndim)
        m = max(1, n // 3)
        b = R.Batch([p, p], [m, n])
        b.launch(R.RunOpts(w.seed, 0, 0))
        first, second = b.read(0), b.read(1)
        b.launch(R.RunOpts(w.seed, 0, 0, 0, 0, 3, 256))
        _same(first, b.read(0), 2 * w.ndim)
        _same(second, b.read(1), 2 * w.ndim)
        _same(first, p.run(m, w.seed), 2 * w.ndim)
    p.close()


@pytest.mark.parametrize("tau0", [1.0e3, 4.0e3, 1.2e4])
def test_moving_grids_of_thin_and_thick_cells_match_the_oracle(tau0):
    # cells of optical depth 250, 1000 and 3000: rows only, and either side of the
    # line between heads and pairs, in launches below, at and past one round
    w = W.Workload(f"cells_{tau0:.0f}", 3, (8, 8, 8), 12, -7.0, 7.0, tau0, 1.0e4, 1, 0x5EED0B06, sphere=True,
                   vmax_kms=40.0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = C.Grid(w)
    ot = g.table()
    p = R.Problem(w)
    thr, _ = p.rows()
    sel = np.repeat(w.mask().astype(bool), w.J)
    ot["thr"][sel] = thr[sel]
    for n in (3000, 800 * sms, 2100 * sms):
        p.reset()
        p.launch(n, w.seed, steps_per_launch=40)
        p.launch(n, w.seed, steps_per_launch=40, resume=1, max_steps=77)
        _same(p.read(), C.walk(g, ot, w.seed, 0, n, max_steps=77), 6)
    p.close()

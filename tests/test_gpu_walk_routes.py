"""Every way the walk reads its transitions, and both register budgets, on either
side of the lines between them: moving, dusty and static grids of thin and thick
cells in launches below, at and past what three and four CTAs per SM hold,
against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import coracle as C  # noqa: E402
from paper_1709_10187_gb300 import build as B  # noqa: E402
from paper_1709_10187_gb300 import rddmc as R  # noqa: E402
from paper_1709_10187_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
SLAB = W.Workload("routes_slab", 1, (8, 1, 1), 12, -6.0, 6.0, 1.0, 1.0e4, 1, 0x5EED0F01)
CUBE = W.Workload("routes_cube", 3, (8, 8, 8), 12, -6.0, 6.0, 1.0, 1.0e4, 1, 0x5EED0F02, sphere=True)


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


# bins one Doppler width wide: the share of frequency moves is the cells' depth
@pytest.mark.parametrize("w,v,dust,depth", [
    (SLAB, 30.0, 0.0, 60.0), (SLAB, 30.0, 0.0, 400.0), (SLAB, 30.0, 0.0, 8.0e4), (SLAB, 0.0, 0.0, 60.0),
    (SLAB, 30.0, 2.0, 60.0), (CUBE, 30.0, 0.0, 300.0), (CUBE, 30.0, 0.0, 4.0e4), (CUBE, 30.0, 0.0, 6.0e4),
    (CUBE, 30.0, 2.0, 700.0), (CUBE, 0.0, 0.0, 60.0), (CUBE, 0.0, 0.0, 150.0), (CUBE, 0.0, 0.0, 4.0e4),
    (CUBE, 0.0, 2.0, 60.0), (CUBE, 0.0, 2.0, 1.0e3), (CUBE, 0.0, 2.0, 6.0e4)],
    ids=lambda x: getattr(x, "name", f"{x:g}" if isinstance(x, float) else str(x)))
def test_walks_match_the_oracle_on_every_route(w, v, dust, depth):
    w = w.with_(tau0=depth * w.n[0] / 2.0, vmax_kms=v)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = C.Grid(w, dust_abs=dust)
    ot = g.table()
    p = R.Problem(w, dust_abs=dust)
    thr, _ = p.rows()
    sel = np.ones(w.ncell * w.J, bool) if w.mask() is None else np.repeat(w.mask().astype(bool), w.J)
    ot["thr"][sel] = thr[sel]  # walk the device's own thresholds (equal to one count)
    for n in (2000, 900 * sms, 1100 * sms):  # below three CTAs of 256, the fourth's, past both
        p.reset()
        p.launch(n, w.seed, steps_per_launch=32)
        p.launch(n, w.seed, steps_per_launch=32, resume=1, max_steps=61)
        got, want = p.read(), C.walk(g, ot, w.seed, 0, n, max_steps=61)
        for k in ("emitted", "escaped", "aborted", "steps", "clamps", "event_draws", "absorbed"):
            assert got[k] == want[k], (n, k)
        assert np.array_equal(got["hist"], want["hist"]) and np.array_equal(got["sb"], want["sb"])
        assert np.array_equal(got["faces"][:2 * w.ndim], want["faces"][:2 * w.ndim])
    p.close()


def test_heads_of_a_large_moving_table_match_slices():
    # 1.7e7 rows: four CTAs per SM however many packets; the slices and an explicit
    # shape walk the same streams
    med = W.clumpy_medium(n=44, J=200, x_max=100.0, tau0=1.0e6, brick=1)
    p, n = R.Problem.clumpy(med), 2000
    assert p.sizes.n_class * p.J > 1 << 24
    a = p.run(n, 5, max_steps=400)
    b = p.run(n, 5, max_steps=400, threads_per_cta=128, ctas_per_sm=2)
    p.reset()
    for k in range(100):
        p.launch(n, 5, steps_per_launch=4, resume=int(k > 0), max_steps=400)
    c = p.read()
    for k in ("emitted", "escaped", "steps", "clamps", "event_draws"):
        assert a[k] == b[k] == c[k], k
    assert np.array_equal(a["hist"], b["hist"]) and np.array_equal(a["hist"], c["hist"])
    p.close()


@pytest.mark.parametrize("w", [W.SMALL.with_(tau0=1.0e4), W.SPHERE8_V, W.SPHERE8], ids=lambda w: w.name)
def test_hybrid_walk_does_not_depend_on_its_register_budget(w):
    # more packets than two CTAs per SM hold take four, with counters in registers;
    # explicit shapes of fewer packets take the two: each packet's walk is its own
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p, n = R.Problem(w, mode=R.MODE_HYBRID), 512 * sms
    big = n + 4096
    keys = ("emitted", "escaped", "steps", "mc_events", "conversions", "event_draws", "clamps")
    whole = p.run(big, w.seed, max_steps=40)
    p.reset()
    p.launch(big, w.seed, steps_per_launch=20, max_steps=40)
    p.launch(big, w.seed, steps_per_launch=20, resume=1, max_steps=40)
    cut = p.read()
    for k in keys:
        assert whole[k] == cut[k], k
    assert np.array_equal(whole["hist"], cut["hist"])
    p.reset()
    p.launch(n, w.seed, steps_per_launch=40)
    few = p.packet_states(n, 0, n)
    p.reset()
    p.launch(big, w.seed, steps_per_launch=40)
    many = p.packet_states(big, 0, n)
    for k in few:
        fly = (few["status"] == 1) & (many["status"] == 1)
        assert np.array_equal(few["status"], many["status"]) and np.array_equal(few[k][fly], many[k][fly]), k
    p.close()


@pytest.mark.parametrize("depth", [60.0, 700.0, 6.0e4])
@pytest.mark.parametrize("moving", [False, True])
def test_batches_match_the_oracle_on_every_route(depth, moving):
    # batches of static cubes (thin and thick) and with a moving grid (pairs, or heads
    # where the packets fill the chip), few packets and more than fit at once
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ws = [CUBE.with_(tau0=depth * 4.0, vmax_kms=30.0 if moving else 0.0),
          SLAB.with_(tau0=depth * 4.0), CUBE.with_(tau0=depth * 4.0, J=9, seed=3)]
    ps, ots, gs = [R.Problem(w) for w in ws], [], []
    for w, p in zip(ws, ps):
        g = C.Grid(w)
        ot = g.table()
        thr, _ = p.rows()
        sel = np.ones(w.ncell * w.J, bool) if w.mask() is None else np.repeat(w.mask().astype(bool), w.J)
        ot["thr"][sel] = thr[sel]
        gs.append(g)
        ots.append(ot)
    for total in (3000, 1100 * sms):
        n = [total // 2, total // 6, total // 3]
        b = R.Batch(ps, n)
        b.launch(R.RunOpts(0x5EED, 0, 45))
        first = 0
        for i, w in enumerate(ws):
            got, want = b.read(i), C.walk(gs[i], ots[i], 0x5EED, first, n[i], max_steps=45)
            for k in ("emitted", "escaped", "aborted", "steps", "clamps", "event_draws"):
                assert got[k] == want[k], (total, i, k)
            assert np.array_equal(got["hist"], want["hist"]) and np.array_equal(got["sb"], want["sb"])
            first += n[i]
    for p in ps:
        p.close()

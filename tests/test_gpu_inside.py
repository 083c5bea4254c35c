"""Cells four moves inside their class, whose transitions the walk takes without
following the class: grids with none, one and a few of them, against the
oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import coracle as C  # noqa: E402
from paper_1709_10187_gb300 import build as B  # noqa: E402
from paper_1709_10187_gb300 import rddmc as R  # noqa: E402
from paper_1709_10187_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


@pytest.mark.parametrize("n", [(8, 1, 1), (9, 1, 1), (10, 1, 1), (11, 1, 1), (9, 9, 9), (11, 10, 12), (21, 9, 8)])
@pytest.mark.parametrize("clump", [False, True])
def test_cells_around_the_middle_match_the_oracle(n, clump):
    # the outermost cells are a class of their own (their faces are exterior), so a
    # uniform axis of eleven cells has one cell four moves inside; a denser cell
    # off the middle cuts the region again
    ndim = 1 if n[1] == 1 else 3
    n_rel = np.ones(n[0] * n[1] * n[2])
    if clump:
        n_rel[n_rel.size // 2 + 3] = 2.5
    w = W.Workload("inside", ndim, n, 13, -40.0, 40.0, 1.5e3, 1.0e4, 4000, 0x5EED0E01)
    g = C.Grid(w, n_rel=n_rel)
    ot = g.table()
    p = R.Problem(w, n_rel=n_rel)
    ot["thr"], _ = p.rows()  # walk the device's own thresholds (equal to one count)
    orc = C.walk(g, ot, w.seed, 0, w.packets, max_steps=1 << 62)
    b = R.Batch([p], [w.packets])
    b.launch(R.RunOpts(w.seed, 0, 0))
    for got in (p.run(w.packets, w.seed), b.read(0)):
        for k in ("emitted", "escaped", "aborted", "steps", "event_draws"):
            assert got[k] == orc[k], k
        assert np.array_equal(got["hist"], orc["hist"]) and np.array_equal(got["faces"][:2 * ndim], orc["faces"][:2 * ndim])
    p.close()

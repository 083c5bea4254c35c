"""Rows of moving grids of few bins, where a block of the table kernel takes
several classes: thresholds against the FP64 oracle at the sizes where a block's
classes change, and the time of small tables against larger ones."""
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


@pytest.mark.parametrize("J", [1, 2, 3, 4, 9, 31, 41, 42, 63, 64])
@pytest.mark.parametrize("ndim,hybrid", [(3, False), (3, True), (1, False)])
def test_moving_rows_of_several_classes_per_block(J, ndim, hybrid):
    # 128 edges: 64, 42, 32, 25 classes of few bins, three of 41, two to J = 63, one from 64
    x = max(4.0, 0.3 * J)
    w = W.SPHERE8_V.with_(name=f"classes_{J}", J=J, x_min=-x, x_max=x)
    if ndim == 1:
        w = W.Workload(f"classes_slab_{J}", 1, (11, 1, 1), J, -x, x, 3.0e3, 1.0e4, 1, 1, vmax_kms=25.0)
    ot = C.Grid(w, hybrid=hybrid).table()
    p = R.Problem(w, mode=R.MODE_HYBRID if hybrid else R.MODE_DDMC)
    thr, flags = p.rows()
    p.close()
    sel = np.ones(w.ncell * J, bool) if w.mask() is None else np.repeat(w.mask().astype(bool), J)
    assert np.array_equal(flags[sel], ot["flags"][sel])
    # one count where CUDA's and the C library's exp/erfc round differently
    d = thr[sel].astype(np.int64) - ot["thr"][sel].astype(np.int64)
    assert np.abs(d).max() <= 1 and (d != 0).sum() <= max(2, 1e-4 * d.size)


def test_tables_of_few_bins_take_less_time():
    # a table's work grows with its edges: 2 bins have 3 of them, 62 have 63
    def ms(J):
        med = W.clumpy_medium(n=32, J=J, x_max=max(4.0, J / 2.0), tau0=1.0e6, brick=1)
        p = R.Problem.clumpy(med)
        best = 1e9
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            a.record()
            R.precompute_leakage(p.grid, p.params, p.table.data_ptr(), p.table.numel(), p.stream())
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        p.close()
        return best

    small, large = ms(2), ms(62)
    assert small < 0.25 * large, (small, large)


@pytest.mark.parametrize("n,J", [(10, 2), (10, 40), (12, 31), (18, 62), (22, 31)])
def test_rows_do_not_depend_on_how_blocks_share_classes(n, J):
    # every cell a class of its own: few classes go one to a block, more fill its
    # threads
    x = max(4.0, J / 2.0)
    w = W.Workload(f"shared_{n}_{J}", 3, (n, n, n), J, -x, x, 1.0e5, 1.0e4, 1, 1, vmax_kms=60.0)
    n_rel = W.clumpy_medium(n=n, J=J, brick=1).n_rel
    ot = C.Grid(w, n_rel=n_rel).table()
    p = R.Problem(w, n_rel=n_rel)
    thr, flags = p.rows()
    assert p.sizes.n_class == w.ncell
    p.close()
    assert np.array_equal(flags, ot["flags"])
    d = thr.astype(np.int64) - ot["thr"].astype(np.int64)
    assert np.abs(d).max() <= 1 and (d != 0).sum() <= max(2, 1e-4 * d.size)

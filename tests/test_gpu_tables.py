"""Table kernels at the sizes where their tiling can go wrong, against the FP64
oracle: the profile kernel takes 31 bins per block, the rows of a moving grid
127 per block, the redistribution sweeps 16 pieces at a time and averages its
nodes over a cluster of up to 8 blocks."""
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


def _check(w, hybrid):
    ot = C.Grid(w, hybrid=hybrid).table()
    p = R.Problem(w, mode=R.MODE_HYBRID if hybrid else R.MODE_DDMC)
    thr, flags = p.rows()
    p.close()
    m = w.mask()
    sel = np.ones(w.ncell * w.J, bool) if m is None else np.repeat(m.astype(bool), w.J)
    assert np.array_equal(flags[sel], ot["flags"][sel])
    # one count where CUDA's and the C library's exp/erfc round differently
    d = thr[sel].astype(np.int64) - ot["thr"][sel].astype(np.int64)
    assert np.abs(d).max() <= 1
    assert (d != 0).sum() <= max(2, 1e-4 * d.size), (d != 0).sum()


@pytest.mark.parametrize("J", [1, 2, 30, 31, 32, 62, 63, 129])
def test_static_rows_at_profile_block_edges(J):
    x = max(4.0, 0.3 * J)
    _check(W.Workload(f"rows_slab_{J}", 1, (7, 1, 1), J, -x, x, 3.0e3, 1.0e4, 1, 1), hybrid=False)


@pytest.mark.parametrize("hybrid", [False, True], ids=["ddmc", "hybrid"])
@pytest.mark.parametrize("J", [2, 126, 127, 128, 254, 255])
def test_moving_rows_at_tile_edges(J, hybrid):
    x = max(4.0, 0.2 * J)
    _check(W.SPHERE8_V.with_(name=f"rows_sphere_{J}", J=J, x_min=-x, x_max=x), hybrid)


def _rule_cdf(edges, xp, a):
    """F(e | x') at the interior edges by the thresholds' quadrature rule, in numpy: x
    pieces between x' - 14 and x' + 14 cut at the integers, the interior edges, x'
    and -x', 16 Gauss-Legendre nodes each; u pieces from |x - x'|/2 over 6, cut at
    max(x, x') and -min(x, x') and 4 a 4^k (k = 0..6) on either side, 8 nodes."""
    g16, g8 = np.polynomial.legendre.leggauss(16), np.polynomial.legendre.leggauss(8)

    def g(x):
        hi, lo = max(x, xp), min(x, xp)
        z0 = 0.5 * abs(x - xp)
        cut = [z0, z0 + 6.0]
        for p in (hi, -lo):
            for d in [0.0] + [s * 4.0 * a * 4.0 ** k for k in range(7) for s in (-1, 1)]:
                if z0 < p + d < z0 + 6.0:
                    cut.append(p + d)
        cut = np.sort(cut)
        h, c = 0.5 * np.diff(cut), 0.5 * (cut[1:] + cut[:-1])
        u = c[:, None] + h[:, None] * g8[0]
        f = np.exp(-u * u) * (np.arctan((lo + u) / a) - np.arctan((hi - u) / a))
        return float((h * (f * g8[1]).sum(1)).sum())

    lo, hi = xp - 14.0, xp + 14.0
    cut = {lo, hi, xp, -xp, *np.arange(np.ceil(lo), hi), *edges[1:-1]}
    cut = np.array(sorted(v for v in cut if lo <= v <= hi))
    h, c = 0.5 * np.diff(cut), 0.5 * (cut[1:] + cut[:-1])
    piece = [hh * sum(w * g(cc + hh * t) for t, w in zip(*g16)) for hh, cc in zip(h, c)]
    cum = np.concatenate([[0.0], np.cumsum(piece)])
    return np.array([cum[np.searchsorted(cut, min(max(v, lo), hi))] for v in edges[1:-1]]) / cum[-1]


@pytest.mark.parametrize("J,n_sub", [(2, 1), (9, 8), (33, 1), (40, 2)])
def test_redistribution_rows_follow_the_rule(J, n_sub):
    w = W.Workload(f"redist_{J}", 1, (3, 1, 1), J, -0.4 * J, 0.4 * J, 100.0, 1.0e4, 1, 1)
    p = R.Problem(w, mode=R.MODE_HYBRID)
    thr = p.redistribution(n_sub).cpu().numpy().view(np.uint32)[: J * (J - 1)].reshape(J, J - 1)
    p.close()
    e = w.edges()
    gx, gw = np.polynomial.legendre.leggauss(n_sub)
    for jp in {0, J // 2, J - 1}:
        c = np.zeros(J - 1)
        for xg, wg in zip(gx, gw):
            xp = 0.5 * (e[jp + 1] - e[jp]) * xg + 0.5 * (e[jp + 1] + e[jp])
            c += 0.5 * wg * _rule_cdf(e, xp, C.damping(w.T))
        # the same rule with its nodes and functions rounded elsewhere: 1e-13
        # relative at most, so a threshold moves by one count where it rounds
        q = np.minimum(np.rint(c * 2.0 ** 32), 2.0 ** 32 - 1)
        assert np.abs(thr[jp].astype(np.float64) - q).max() <= 1, jp

"""Cell binning, neighbor lists and the feasibility check of the standalone calls at the edges of
their two forms (one block per instance up to 2048 circles, tiles of 256 circles beyond), against the
oracle (marked gpu).  Cells, order, lists and depths are those of correctly rounded operations: the
kernels search in binary32 and decide in binary64 what that cannot, so everything is compared bit
for bit."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2303_02650_gb300 import synth
from gpu_util import need_gpu, split

pytestmark = pytest.mark.gpu

SIZES = {"small": [1, 64, 65, 0, 2047, 2048, 256], "large": [2049, 2304, 2305, 9000], "both": [700, 5000, 3, 2048, 2600]}


def _layout(n, R, seed, kind):
    rng = np.random.default_rng(seed)
    parts = []
    for nq, Rq in zip(n, R):
        x = synth.random_layout(int(nq), 0.9 * float(Rq), seed + int(nq))
        if kind == "clusters" and nq > 60:  # rows past the 16 hits a lane keeps, coincident circles, far ones
            x[:40] = x[50] + rng.normal(scale=0.3, size=(40, 2))
            x[41] = x[42]
            x[43] = (3.0 * Rq, -2.5 * Rq)
            x[44:48] += 1e5
        if kind == "grid":  # circles on the cells' edges and pairs at the cutoff
            x = np.round(x / 1.25) * 1.25
        parts.append(x)
    return np.concatenate(parts) if parts else np.zeros((0, 2))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("sizes", list(SIZES))
@pytest.mark.parametrize("kind,u", [("plain", 0.83), ("clusters", 0.83), ("grid", 0.83), ("plain", 0.02)])
def test_cells_lists_and_depths(orc, prec, sizes, kind, u):
    torch, pecc = need_gpu()
    n = np.array(SIZES[sizes], dtype=np.int32)
    R = np.array([synth.radius(max(int(v), 1), u) for v in n])
    xy = _layout(n, R, 11, kind)
    # a capacity that holds the crowded layouts
    with pecc.Context(n, precision=prec, nbr_capacity=64.0) as c:
        c.set_radius(R)
        c.set_positions(torch.from_numpy(xy))
        xy = c.get_positions().cpu().numpy()
        assert c.rebuild_neighbors(force=True).cpu().numpy().all()
        key, order = [t.cpu().numpy() for t in c.export_cells()]
        rp, col = [t.cpu().numpy() for t in c.export_neighbors()]
        feas, mo = [t.cpu().numpy() for t in c.check_feasible()]
        again = c.rebuild_neighbors(force=False).cpu().numpy()
        # one circle of every second instance moves past the displacement rule
        off = np.concatenate([[0], np.cumsum(n)])
        moved = xy.copy()
        pick = np.array([q % 2 == 0 and n[q] > 0 for q in range(len(n))])
        for q in np.nonzero(pick)[0]:
            moved[off[q + 1] - 1, 0] += 0.26
        c.set_positions(torch.from_numpy(moved))
        third = c.rebuild_neighbors(force=False).cpu().numpy()
    assert not again.any()
    assert np.array_equal(third.astype(bool), pick)
    for q in range(len(n)):
        a, b = off[q], off[q + 1]
        kref = orc.cell_keys(xy[a:b], float(R[q]), 2.5)
        assert np.array_equal(key[a:b].astype(np.uint32), kref), q
        assert np.array_equal(order[a:b], np.argsort(kref, kind="stable")), q
        rref, cref = orc.neighbors_brute(xy[a:b], 2.5, prec32=(prec == 1))
        assert np.array_equal(rp[a:b + 1] - rp[a], rref), q
        assert np.array_equal(col[rp[a]:rp[b]] - a, cref), q
        ref = orc.max_overlap(xy[a:b], float(R[q]))[0] if n[q] else 0.0
        assert mo[q] == ref and feas[q] == (1 if ref <= 1e-9 else 0), q


@pytest.mark.parametrize("sizes", list(SIZES))
def test_check_nonfinite_overflow_and_near_contact(orc, sizes):
    """NaN where an instance cannot be checked, its neighbors unaffected; the deepest pair of an
    almost touching lattice (depths within binary32 rounding of each other) exactly."""
    torch, pecc = need_gpu()
    n = np.array([v for v in SIZES[sizes] if v > 60], dtype=np.int32)
    R = np.array([2.2 * np.sqrt(float(v)) for v in n])
    rng = np.random.default_rng(5)
    parts = []
    for v in n:
        side = int(np.ceil(np.sqrt(v)))
        ij = np.stack(np.meshgrid(np.arange(side), np.arange(side)), -1).reshape(-1, 2)[:v]
        parts.append((ij - side / 2) * (2.0 - 1e-10) + rng.uniform(-1e-12, 1e-12, size=(v, 2)))
    xy = np.concatenate(parts)
    off = np.concatenate([[0], np.cumsum(n)])
    bad, full = 0, 1 if len(n) > 1 else 0
    xy2 = xy.copy()
    xy2[off[bad] + 3, 1] = np.nan
    if full != bad:
        xy2[off[full]:off[full + 1]] = 0.25  # every pair a neighbor: past any capacity
    with pecc.Context(n, precision=0) as c:
        c.set_radius(R)
        c.set_positions(torch.from_numpy(xy))
        feas, mo = [t.cpu().numpy() for t in c.check_feasible(1e-9)]
        c.set_positions(torch.from_numpy(xy2))
        feas2, mo2 = [t.cpu().numpy() for t in c.check_feasible(1e-9)]
    for q, x in enumerate(split(xy, n)):
        ref = orc.max_overlap(x, float(R[q]))[0]
        assert mo[q] == ref and feas[q] == (1 if ref <= 1e-9 else 0), q
        if q in (bad, full):
            assert np.isnan(mo2[q]) and feas2[q] == 0
        else:
            assert mo2[q] == ref


@pytest.mark.parametrize("sizes", [[1, 64, 65, 2047, 2048], [2049, 2305], [300, 2600, 0, 12]])
@pytest.mark.parametrize("kind,u", [("plain", 0.83), ("clusters", 0.83), ("grid", 0.83), ("plain", 0.02)])
def test_features_at_the_edges(sizes, kind, u):
    """The 25 features bit for bit: full and short rows, more than 32 circles within 4.5 (the buffer
    of a lane is emptied on the way), equal distances (index order), coincident circles."""
    torch, pecc = need_gpu()
    n = np.array(sizes, dtype=np.int32)
    R = np.array([synth.radius(max(int(v), 1), u) for v in n])
    xy = _layout(n, R, 23, kind)
    with pecc.Context(n, precision=1) as c:
        c.set_radius(R)
        c.set_positions(torch.from_numpy(xy))
        xy = c.get_positions().cpu().numpy().astype(np.float32)
        f = c.features().cpu().numpy()
    for q, (fq, xq) in enumerate(zip(split(f, n), split(xy, n))):
        if n[q]:
            assert np.array_equal(fq, omlp.features(xq, float(R[q]))), q

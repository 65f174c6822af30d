"""Calls at the limits of what they take (marked gpu): list overflow of any length, shared memory of any
size, contexts of several host threads, waits that run out, radii that are not radii or past binary32's
range, cutoffs close to 2, circles in one place or crowded."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2303_02650_gb300 import synth
from gpu_util import need_gpu, split

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("prec", [0, 1])
def test_overflow_past_32_bit_counts(orc, prec):
    """50000 circles in one place: 2.5e9 list entries, more than a 32-bit count holds.  Lists, energy and
    check report the overflow; the instance beside them is unaffected."""
    torch, pecc = need_gpu()
    n = np.array([50000, 300], dtype=np.int32)
    R = np.array([synth.radius(int(v), 0.8) for v in n])
    x = synth.random_layout(300, 0.9 * float(R[1]), 3).astype(np.float32).astype(np.float64)
    with pecc.Context(n, precision=prec) as c:
        c.set_radius(R)
        c.set_positions(torch.from_numpy(np.concatenate([np.zeros((50000, 2)), x])))
        assert c.rebuild_neighbors(force=True).cpu().numpy().all()
        with pytest.raises(pecc.PeccError, match="NBR_OVERFLOW"):
            c.export_neighbors()
        E, g = [t.cpu().numpy() for t in c.energy_grad()]
        feas, mo = [t.cpu().numpy() for t in c.check_feasible()]
    assert np.isnan(E[0]) and np.isnan(g[:50000]).all()
    assert np.isfinite(E[1]) and np.isfinite(g[50000:]).all()
    assert np.isnan(mo[0]) and mo[1] == orc.max_overlap(x, float(R[1]))[0] and feas[0] == 0


def test_whole_gpu_overflow_past_32_bit_counts():
    """600000 circles closer than the cutoff to one another: a block's share of the rows (3948 of them, each
    with 599999 entries) passes 32 bits.  The descent ends with the overflow status."""
    torch, pecc = need_gpu()
    n = 600000
    rng = np.random.default_rng(1)
    r, a = 0.6 * np.sqrt(rng.uniform(size=n)), rng.uniform(0.0, 2.0 * np.pi, size=n)
    with pecc.Context(np.array([n], dtype=np.int32), precision=1, max_iter=1) as c:
        c.set_radius(np.array([synth.radius(n, 0.8)]))
        c.set_positions(torch.from_numpy(np.stack([r * np.cos(a), r * np.sin(a)], 1)))
        iters, status = c.descend()
        assert int(status.cpu()[0]) == 4 and int(iters.cpu()[0]) == 0


# The first call of a process: nothing has raised a kernel's shared-memory limit before it.
FIRST_CALL = """
import sys
import numpy as np, torch
import oracle as orc
from oracle import mlp as omlp
from paper_2303_02650_gb300 import pecc, synth
kind, n0, others, prec = sys.argv[1], int(sys.argv[2]), int(sys.argv[3]), int(sys.argv[4])
orc.build()
n = np.array([n0] + [1] * others, dtype=np.int32)
R = np.array([synth.radius(int(v), 0.8) for v in n])
x = synth.random_layout(n0, 0.9 * float(R[0]), 3).astype(np.float32).astype(np.float64)
xy = np.concatenate([x, np.zeros((others, 2))])
with pecc.Context(n, precision=prec) as c:
    c.set_radius(R)
    c.set_positions(torch.from_numpy(xy))
    if kind == "check":
        assert float(c.check_feasible()[1][0]) == orc.max_overlap(x, float(R[0]))[0]
    elif kind == "features":
        assert np.array_equal(c.features().cpu().numpy()[:n0], omlp.features(x.astype(np.float32), float(R[0])))
    else:
        c.rebuild_neighbors(force=True)
        if kind == "lists":
            rp, col = [t.cpu().numpy() for t in c.export_neighbors()]
            rref, cref = orc.neighbors_brute(x, 2.5, prec32=(prec == 1))
            assert np.array_equal(rp[:n0 + 1], rref) and np.array_equal(col[:rp[n0]], cref)
        else:
            E, g = c.energy_grad()
            torch.cuda.synchronize()
            assert np.isfinite(E.cpu().numpy()).all() and bool(torch.isfinite(g).all())
print("first call ok")
"""


@pytest.mark.parametrize("kind,n,others,prec", [
    ("check", 1790, 0, 0), ("check", 1790, 0, 2), ("lists", 1706, 0, 1), ("lists", 1200, 0, 0), ("lists", 1503, 200, 0),
    ("features", 1218, 0, 1), ("energy", 6136, 0, 1), ("energy", 3064, 0, 0)])
def test_first_call_of_a_process(orc, kind, n, others, prec):
    """Sizes whose dynamic shared memory is just below 48 KB, and above it with the kernel's own."""
    need_gpu()
    r = subprocess.run([sys.executable, "-c", FIRST_CALL, kind, str(n), str(others), str(prec)], cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "first call ok" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]


def test_contexts_of_two_host_threads():
    """Two threads whose contexts need different amounts of shared memory, each on its own stream, launching
    without pause: every call of both succeeds with the results it has alone."""
    torch, pecc = need_gpu()
    sizes, rounds = [1900, 2048], 1500
    errors, got = [], {}

    def work(n0, gate=None, out=got):
        try:
            s = torch.cuda.Stream()
            R = np.array([synth.radius(n0, 0.8)])
            x = torch.from_numpy(synth.random_layout(n0, 0.9 * float(R[0]), 3))
            with torch.cuda.stream(s), pecc.Context(np.array([n0], dtype=np.int32), precision=1, stream=s) as c:
                m = pecc.MLP(7, stream=s)
                c.set_radius(R)
                c.set_positions(x)
                s.synchronize()
                if gate:
                    gate.wait()
                c.warm_start(m, rounds)  # list builds, energies and features, enqueued by one call
                mo = c.check_feasible()[1]
                xy = c.get_positions()
                s.synchronize()
                out[n0] = np.concatenate([xy.cpu().numpy().ravel(), mo.cpu().numpy()])
                m.close()
        except Exception as e:  # noqa: BLE001 -- reported by the test's own thread
            errors.append((n0, repr(e)))
            if gate:
                gate.abort()

    alone = {}
    for v in sizes:
        work(v, out=alone)
    gate = threading.Barrier(len(sizes))
    threads = [threading.Thread(target=work, args=(v, gate)) for v in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for v in sizes:
        assert np.array_equal(got[v], alone[v])


@pytest.mark.parametrize("short_lanes,yes", [(0, 32), (1, 0), (0x80000000, 0), (0x55555555, 0), (0xFFFFFFFF, 0)])
def test_a_warp_has_one_answer_to_a_wait(short_lanes, yes):
    """A wait for the tensor cores that runs out in some lanes of a warp and not in others: all of them
    hear that it ran out (warp-wide instructions follow)."""
    torch, pecc = need_gpu()
    assert pecc.selftest_mma_wait(200_000_000, short_lanes) == yes


def _apart(n):
    """Layouts of circles that do not overlap: squares of side 2.5."""
    parts = []
    for v in n:
        side = int(np.ceil(np.sqrt(v)))
        g = np.stack(np.meshgrid(np.arange(side), np.arange(side)), -1).reshape(-1, 2)[:v] * 2.5
        parts.append(g - g.mean(0) if v else g.astype(float))
    return np.concatenate(parts).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("bad", [-1.0, 0.0, float("nan"), float("inf")])
def test_rejected_radius_is_reported(orc, bad):
    """Circles that do not overlap, in containers whose radius is not finite and > 0: not checkable, no energy,
    no descent, in the block, tile, whole-GPU and explicit-Hessian forms; the instances beside them are
    unaffected, and one without circles has nothing to report."""
    torch, pecc = need_gpu()
    n = np.array([7, 7000, 30, 0, 16500], dtype=np.int32)
    off = np.concatenate([[0], np.cumsum(n)])
    xy = _apart(n)
    R = np.array([bad, bad, 12.0, bad, bad])
    for prec in (0, 1, 2):
        with pecc.Context(n, precision=prec) as c:
            c.set_radius(R)
            c.set_positions(torch.from_numpy(xy))
            feas, mo = [t.cpu().numpy() for t in c.check_feasible()]
            c.rebuild_neighbors(force=True)
            E, g = [t.cpu().numpy() for t in c.energy_grad()]
            status = c.descend()[1].cpu().numpy()
            x1 = c.get_positions().cpu().numpy()
            assert np.array_equal(c.check_feasible()[0].cpu().numpy(), feas)
        assert feas.tolist() == [0, 0, 1, 1, 0] and np.isnan(mo[[0, 1, 4]]).all()
        x2 = xy[off[2]:off[3]]
        assert mo[2] == orc.max_overlap(x2, 12.0)[0] and mo[3] == 0.0
        for q in (0, 1, 4):
            assert np.isnan(E[q]) and np.isnan(g[off[q]:off[q + 1]]).all() and status[q] == 5
            assert np.array_equal(x1[off[q]:off[q + 1]], xy[off[q]:off[q + 1]])
        assert E[2] == 0.0 and not g[off[2]:off[3]].any() and E[3] == 0.0 and status[[2, 3]].tolist() == [0, 0]
    n = n[:4]
    with pecc.Context(n, precision=0, qn_dense=1) as c:
        c.set_radius(R[:4])
        c.set_positions(torch.from_numpy(xy[:off[4]]))
        assert c.descend()[1].cpu().numpy().tolist() == [5, 5, 0, 0]


@pytest.mark.parametrize("l_cut", [2.05, 2.1, 2.249, 2.25, 3.0])
def test_features_reach_over_small_cells(l_cut):
    """Cells of side l_cut: every circle within 4.5 is found, also where 4.5 spans three cells."""
    torch, pecc = need_gpu()
    n = np.array([900, 2600], dtype=np.int32)
    R = np.array([synth.radius(int(v), 0.3) for v in n])  # about six circles within 4.5: all are kept
    xy = np.concatenate([synth.random_layout(int(v), float(r), 31 + int(v)) for v, r in zip(n, R)])
    half = (l_cut - 2.0) / 2.0
    with pecc.Context(n, precision=1, l_cut=l_cut, rebuild_disp=half, step_max=half) as c:
        c.set_radius(R)
        c.set_positions(torch.from_numpy(xy))
        xy = c.get_positions().cpu().numpy().astype(np.float32)
        f = c.features().cpu().numpy()
    for q, (fq, xq) in enumerate(zip(split(f, n), split(xy, n))):
        assert np.array_equal(fq, omlp.features(xq, float(R[q]))), q


@pytest.mark.parametrize("R0", [1e36, 1e37, 2e38, 1e39, 1e100])
def test_cells_of_huge_containers(orc, R0):
    """Radii near and past the largest binary32 value: the cells are those of the binary64 operations."""
    torch, pecc = need_gpu()
    n = np.array([300, 2100], dtype=np.int32)
    R = np.array([R0, R0])
    xy = np.concatenate([synth.random_layout(int(v), R0, 5 + int(v)) for v in n])
    xy[:4] = [[0.5, -0.5], [0.5, 1.5], [-R0, R0], [3.0 * R0, 0.0]]
    with pecc.Context(n, precision=0) as c:
        c.set_radius(R)
        c.set_positions(torch.from_numpy(xy))
        c.rebuild_neighbors(force=True)
        key, order = [t.cpu().numpy() for t in c.export_cells()]
        rp, col = [t.cpu().numpy() for t in c.export_neighbors()]
        mo = c.check_feasible()[1].cpu().numpy()
    off = np.concatenate([[0], np.cumsum(n)])
    for q in range(len(n)):
        a, b = off[q], off[q + 1]
        kref = orc.cell_keys(xy[a:b], R0, 2.5)
        assert np.array_equal(key[a:b].astype(np.uint32), kref), q
        assert np.array_equal(order[a:b], np.argsort(kref, kind="stable")), q
        rref, cref = orc.neighbors_brute(xy[a:b], 2.5)
        assert np.array_equal(rp[a:b + 1] - rp[a], rref) and np.array_equal(col[rp[a]:rp[b]] - a, cref), q
        assert mo[q] == orc.max_overlap(xy[a:b], R0)[0], q


@pytest.mark.parametrize("n,R0,expect", [(50000, 260.0, 4), (20000, -1.0, 5), (16384, 1.0, 4)])
def test_whole_gpu_descent_of_coincident_circles(n, R0, expect):
    """All circles in one place (as pecc_init_random leaves them for R <= 1 or a rejected radius): equal
    partition keys, one bucket.  The descent ends with its status well before a barrier's time limit."""
    torch, pecc = need_gpu()
    with pecc.Context(np.array([n], dtype=np.int32), precision=2) as c:
        c.set_radius(np.array([R0]))
        c.init_random(3) if R0 <= 1.0 else c.set_positions(torch.zeros(n, 2, dtype=torch.float64))
        x0 = c.get_positions()
        assert not x0.any()
        iters, status = c.descend()
        assert int(status.cpu()[0]) == expect and int(iters.cpu()[0]) == 0
        assert torch.equal(c.get_positions(), x0)


@pytest.mark.parametrize("prec", [0, 1])
def test_overflow_of_crowded_cells(orc, prec):
    """Crowds around the corner of four cells: the lists overflow, and the crowd's rows (every other circle
    of it, from several cells) are not put in order first.  The rest of the batch is unaffected; a crowd
    that fits is listed in full."""
    torch, pecc = need_gpu()
    n = np.array([2048, 50000, 300, 2048, 3000], dtype=np.int32)
    crowd = [2048, 50000, 0, 120, 150]
    R = np.array([synth.radius(int(v), 0.8) for v in n])
    rng = np.random.default_rng(4)
    parts = []
    for v, m, r in zip(n, crowd, R):
        x = synth.random_layout(int(v), 0.9 * float(r), 3 + int(v))
        side = 2.5 * (1.0 + 2.0 ** -20)
        corner = -r + side * np.floor(r / side)
        x[:m] = corner + rng.uniform(-0.4, 0.4, size=(m, 2))
        parts.append(x.astype(np.float32).astype(np.float64))
    off = np.concatenate([[0], np.cumsum(n)])
    with pecc.Context(n, precision=prec) as c:
        c.set_radius(R)
        c.set_positions(torch.from_numpy(np.concatenate(parts)))
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        c.check_feasible()
        ev[0].record()
        c.rebuild_neighbors(force=True)
        ev[1].record()
        torch.cuda.synchronize()
        assert ev[0].elapsed_time(ev[1]) < 2000.0
        with pytest.raises(pecc.PeccError, match="NBR_OVERFLOW"):
            c.export_neighbors()
        E, g = [t.cpu().numpy() for t in c.energy_grad()]
    for q in range(len(n)):
        if crowd[q] == n[q]:
            assert np.isnan(E[q]) and np.isnan(g[off[q]:off[q + 1]]).all()
        else:
            # binary32: a thread adds up at most about 2400 positive terms, 2^-24 each
            ref = orc.energy_allpairs(parts[q], float(R[q]))
            assert abs(E[q] - ref) <= (1e-12 if prec == 0 else 2e-4) * ref
    keep = [2, 3, 4]
    with pecc.Context(n[keep], precision=prec) as c:
        c.set_radius(R[keep])
        c.set_positions(torch.from_numpy(np.concatenate([parts[q] for q in keep])))
        c.rebuild_neighbors(force=True)
        rp, col = [t.cpu().numpy() for t in c.export_neighbors()]
    a = 0
    for q in keep:
        b = a + n[q]
        rref, cref = orc.neighbors_brute(parts[q], 2.5, prec32=(prec == 1))
        assert np.array_equal(rp[a:b + 1] - rp[a], rref) and np.array_equal(col[rp[a]:rp[b]] - a, cref), q
        a = b

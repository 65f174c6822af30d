"""The descent and the adjustment at the edges of their forms (marked gpu): the secant slots' groups
of six, arrays on chip or in global memory, a line search with and without room for its energy
entries, the adjustment's vector in registers or in memory.

Against the oracle the tolerance is its own sensitivity to rounding: ten times the largest deviation of
oracle runs whose start is perturbed by the arithmetic's relative rounding (and a floor where that is
smaller); equal forms are compared bit for bit."""
import numpy as np
import pytest

from paper_2303_02650_gb300 import synth
from gpu_util import need_gpu, split

pytestmark = pytest.mark.gpu


def _hex(rings, seed):
    """A compressed hexagonal patch: every circle in contact with its neighbors, a smooth descent."""
    x = synth.hex_patch(rings, 1.95)
    rng = np.random.default_rng(seed)
    return x + rng.uniform(-0.01, 0.01, size=x.shape), 1.95 * rings + 0.97


def _envelope(orc, x0, R, trials=4, **kw):
    r = orc.gbo(x0, R, **kw)
    rng = np.random.default_rng(7)
    dev = 0.0
    for _ in range(trials):
        p = orc.gbo(x0 * (1.0 + 1e-15 * rng.standard_normal(x0.shape)), R, **kw)
        dev = max(dev, float(np.abs(p.x - r.x).max()))
    return r, dev


@pytest.mark.parametrize("m", [1, 5, 6, 10])
@pytest.mark.parametrize("k", [1, 2])
def test_memory_sizes_follow_the_oracle(orc, m, k):
    """Enough sweeps that every slot is filled and the oldest evicted, in one and in two groups of
    slots."""
    torch, pecc = need_gpu()
    sweeps = m + 4
    starts = [_hex(rings, 3 + rings) for rings in (2, 5, 9)]
    n = np.array([x.shape[0] for x, _ in starts], dtype=np.int32)
    R = np.array([r for _, r in starts])
    with pecc.Context(n, precision=0, k_batches=k, lbfgs_m=m, max_iter=sweeps) as c:
        c.set_radius(R)
        c.set_positions(torch.from_numpy(np.concatenate([x for x, _ in starts])))
        iters, _ = c.descend()
        x1 = c.get_positions().cpu().numpy()
    for q, b in enumerate(split(x1, n)):
        r, dev = _envelope(orc, starts[q][0], float(R[q]), k=k, m=m, max_iter=sweeps)
        assert int(iters.cpu()[q]) == r.iters
        assert float(np.abs(b - r.x).max()) <= 10.0 * dev + 1e-12, (q, dev)


@pytest.mark.parametrize("m", [5, 10])
def test_whole_gpu_memory_sizes_follow_the_oracle(orc, m):
    torch, pecc = need_gpu()
    x0, R = _hex(74, 1)  # 16651 circles
    sweeps = m + 2
    with pecc.Context(np.array([x0.shape[0]], dtype=np.int32), precision=0, k_batches=2, lbfgs_m=m,
                      max_iter=sweeps) as c:
        c.set_radius(np.array([R]))
        c.set_positions(torch.from_numpy(x0))
        iters, _ = c.descend()
        x1 = c.get_positions().cpu().numpy()
    r, dev = _envelope(orc, x0, R, trials=2, k=2, m=m, max_iter=sweeps)
    assert int(iters.cpu()[0]) == r.iters
    assert float(np.abs(x1 - r.x).max()) <= 10.0 * dev + 1e-12, dev


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("k,m", [(1, 5), (2, 6), (3, 10)])
def test_on_chip_and_spilled_arrays_give_the_same_descent(prec, k, m):
    """The block's whole share of the SM against 8 KB of it: other arrays in global memory, no room
    for the energy entries of a line search.  120 sweeps, jammed instances with long line searches
    among them."""
    torch, pecc = need_gpu()
    n = np.array([1, 2, 7, 50, 64, 65, 130, 700], dtype=np.int32)
    R = np.array([synth.radius(int(v), 0.84) for v in n]) + 0.2
    out = []
    for smem in (0, 8192):
        with pecc.Context(n, precision=prec, k_batches=k, lbfgs_m=m, max_iter=120, stall_window=0,
                          block_threads=128, smem_per_block=smem) as c:
            c.set_radius(R)
            c.init_random(5)
            c.descend()
            out.append((c.get_positions().cpu().numpy(), c.get_stats().cpu().numpy(), c.get_energy().cpu().numpy()))
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("n", [1, 33, 64])
def test_small_binary64_instance_on_two_and_four_warps(n):
    """The default launch of a small binary64 instance (128 threads) against 64 threads."""
    torch, pecc = need_gpu()
    R = np.array([synth.radius(n, 0.8) if n > 1 else 1.5])
    out = []
    for threads in (0, 64):
        with pecc.Context(np.array([n], dtype=np.int32), precision=0, max_iter=300, block_threads=threads) as c:
            c.set_radius(R)
            c.init_random(2)
            c.descend()
            out.append((c.get_positions().cpu().numpy(), c.get_stats().cpu().numpy()))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [1024, 1025])
def test_adjustment_vector_in_registers_and_in_memory(orc, n):
    """The mixed form with the two-loop's vector in registers (to 1024 circles) and in memory."""
    torch, pecc = need_gpu()
    R = float(synth.radius(n, 0.86))
    x0 = orc.init_positions(n, R, 77)
    kw = dict(lambda0=0.05, rounds=2, max_iter=6)
    with pecc.Context(np.array([n], dtype=np.int32), precision=2, max_iter=6) as c:
        c.set_radius(np.array([R]))
        c.set_positions(torch.from_numpy(x0))
        Rs, iters, _ = c.adjust_container(np.array([R]), lambda0=0.05, rounds=2)
        x = c.get_positions().cpu().numpy()
    xr, Rr, res = orc.adjust_container(x0, R, **kw)
    rng = np.random.default_rng(11)
    dR = dx = 0.0
    for _ in range(3):
        xp, Rp, _ = orc.adjust_container(x0 * (1.0 + 1e-7 * rng.standard_normal(x0.shape)), R, **kw)
        dR, dx = max(dR, abs(Rp - Rr)), max(dx, float(np.abs(xp - xr).max()))
    assert int(iters.cpu()[0]) == res.iters
    assert abs(float(Rs.cpu()[0]) - Rr) <= 10.0 * dR + 1e-8 * R
    assert float(np.abs(x - xr).max()) <= 10.0 * dx + 1e-8 * R

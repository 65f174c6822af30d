"""Calls at the limits of what they take (marked gpu): list overflow of any length."""
import numpy as np
import pytest

from paper_2303_02650_gb300 import synth
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


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

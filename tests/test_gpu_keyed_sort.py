"""A step that keys the next sort and the step that sorts by those keys, in the small
blocks of a context with few slots and in the large ones of one with many: no electron
is lost or doubled, and both follow the same electrons."""
import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

from parity import PKEYS, by_id

pytestmark = pytest.mark.gpu

MANY = 2_400_000  # slots beyond the line in both precisions


@pytest.mark.parametrize("precision,tol", [(hpic.HPIC_FP64, 1e-9), (hpic.HPIC_FP32_MIXED, 1e-5)])
@pytest.mark.parametrize("interval", [2, 5])
@pytest.mark.parametrize("n", [33, 20_011])
def test_keyed_then_sorted(precision, tol, interval, n):
    t = W.target(n=(12, 10, 14))
    run = W.run(seed=5, max_history=2)
    rng = np.random.default_rng(n)
    p = {k: rng.uniform(1, t[m] - 1, n) * t["dx"] for k, m in zip("xyz", ("nx", "ny", "nz"))}
    p.update({k: rng.normal(size=n) * 5 for k in ("ux", "uy", "uz")})
    p["tau"] = rng.exponential(0.02, n)
    p["id"] = np.arange(n, dtype=np.uint32)
    tiles, out = [], []
    for many in (False, True):
        s = hpic.Sim(t, W.laser(t, n_macro=0, spot_r=1e-6), run, precision=precision, sort_interval=interval)
        if many:
            s.set_particles({k: np.resize(v, MANY) for k, v in p.items()} | {"id": np.arange(MANY, dtype=np.uint32)})
        s.set_particles(p)
        s.set_clock(interval - 2, n)
        s.step(2)  # the first keys, the second sorts
        got = s.particles()
        assert np.unique(got["id"]).size == len(got["id"]) and n - len(got["id"]) <= 0.1 * n
        tiles.append([tuple((got[k] / t["dx"] // 4).astype(int)) for k in "zyx"])
        out.append(by_id(got))
        s.close()
    a, b = out
    assert np.array_equal(a["id"], b["id"])
    for k in PKEYS:
        assert np.max(np.abs(a[k] - b[k])) <= tol * np.max(np.abs(b[k])), k
    # sorted by tiles some steps ahead: the same tiles at the same places, but for those
    # whose electrons of one key lie in another order across a tile's face
    same = np.mean([np.mean(np.array(x) == np.array(y)) for x, y in zip(*tiles)])
    assert same > 0.8, same

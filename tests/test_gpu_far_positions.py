"""In the unbounded medium an electron may be anywhere: outside the grid it meets the
solid of the nearest cell, however far out it is."""
import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PHYSICS = hpic.HPIC_DRAG | hpic.HPIC_SCATTER | hpic.HPIC_BREM | hpic.HPIC_UNBOUNDED | hpic.HPIC_FSIGMA


@pytest.mark.parametrize("precision", [hpic.HPIC_FP32_MIXED, hpic.HPIC_FP64])
@pytest.mark.parametrize("interval", [0, 2])
@pytest.mark.parametrize("axis", "xyz")
def test_far_electrons_meet_the_nearest_cell(precision, interval, axis):
    t = W.target(n=(9, 7, 8), material="Al")
    run = W.run(seed=2, physics=PHYSICS, max_history=2)
    cells = {"x": 9, "y": 7, "z": 8}
    places = [-0.5, -3.0, 2.0**31 + 3.5, 2.0**32 + 2.5, 3 * 2.0**32 + 1.5, 2.0**53, -2.0**23 - 4, -2.0**33, 2.0**60, -2.0**60]
    n = len(places)
    near = {k: np.full(n, 4.5) for k in "xyz"}
    near[axis] = np.array([0.5 if p < 0 else cells[axis] - 0.5 for p in places])
    far = dict(near, **{axis: np.array(places)})
    Ti = 1e4 * (1 + np.arange(9 * 7 * 8))  # another F_sigma in every cell
    out = []
    for at in (near, far):
        s = hpic.Sim(t, None, run, precision=precision, sort_interval=interval)
        s.set_grid("Ti", Ti)
        p = {k: at[k] * t["dx"] for k in "xyz"}
        p.update(ux=np.full(n, 9.0), uy=np.full(n, 2.0), uz=np.full(n, -3.0), tau=np.full(n, 0.01), id=np.arange(n, dtype=np.uint32))
        s.set_particles(p)
        s.step(1)
        got = s.particles()
        out.append({k: got[k][np.argsort(got["id"])] for k in ("id", "tau", "ux", "uy", "uz")})
        s.step(1)  # with interval 2 this one sorts by the keys of the first
        assert sorted(s.particles()["id"]) == list(range(n))
        s.close()
    a, b = out
    assert np.all(a["tau"] < 0.01)
    for k in a:
        assert np.array_equal(a[k], b[k]), k

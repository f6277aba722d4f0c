"""Few slots are pushed in small blocks, many in large ones: the same electrons
in a context that holds few slots and in one that once held many, in every kind
of step (plain, keying the next sort, sorting, unbounded) and with ragged counts.

From a target at rest one step's electrons do not depend on the order of any sum,
so they agree to the bit; a node of the grid sums some hundred deposits whose
magnitudes add to about ten times the largest current: 1e2 * 10 roundings at most."""
import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

from parity import PKEYS, assert_field_close, assert_vector_close, by_id

pytestmark = pytest.mark.gpu

MANY = 2_400_000  # slots beyond the line in every precision and mode


@pytest.mark.parametrize("precision,tol", [(hpic.HPIC_FP64, 1e-12), (hpic.HPIC_FP32_MIXED, 6e-5)])
@pytest.mark.parametrize("physics,interval", [(63, 0), (63, 1), (63, 2), (63, 5), (1 | 2 | 4 | 64, 0)])
@pytest.mark.parametrize("n,material", [(33, ["C", "H"]), (20_011, ["Au"])])
def test_few_and_many_slots(precision, tol, physics, interval, n, material):
    t = W.compound([(m, None) for m in material], n=(12, 10, 14))
    run = W.run(seed=5, physics=physics, max_history=2)
    rng = np.random.default_rng(n)
    p = {k: rng.uniform(1, t[m] - 1, n) * t["dx"] for k, m in zip("xyz", ("nx", "ny", "nz"))}
    p.update({k: rng.normal(size=n) * 5 for k in ("ux", "uy", "uz")})
    p["tau"] = rng.exponential(0.02, n)
    p["id"] = np.arange(n, dtype=np.uint32)
    out = []
    for many in (False, True):
        s = hpic.Sim(t, W.laser(t, n_macro=0, spot_r=1e-6), run, precision=precision, sort_interval=interval)
        if many:
            s.set_particles({k: np.resize(v, MANY) for k, v in p.items()} | {"id": np.arange(MANY, dtype=np.uint32)})
        s.set_particles(p)
        s.set_clock(3, n)
        s.step(1)
        out.append(s)
    few, many = out
    a, b = by_id(few.particles()), by_id(many.particles())
    assert all(np.array_equal(a[k], b[k]) for k in PKEYS + ("id",))
    if physics == 63:
        assert_vector_close(few.grid, many.grid, "j", tol)
        assert_field_close(few.grid("heat"), many.grid("heat"), tol, "heat")
    ta, tb = few.tallies(), many.tallies()
    for k in tb:
        assert np.allclose(ta[k], tb[k], rtol=1e-6 if precision == hpic.HPIC_FP32_MIXED else 1e-12, atol=0), k
    for s in out:
        s.close()

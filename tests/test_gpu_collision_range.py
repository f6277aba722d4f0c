"""Drag, scatter and emission of one step over the whole range of energies
(small and large deflections, the photon threshold, the tracking cut), in the
box and in the unbounded medium, with ragged electron counts."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

from parity import assert_particles_close, by_id

pytestmark = pytest.mark.gpu


# FP32 from 50 keV up: below, the explicit drag takes most of an electron's energy in
# one step and its remainder loses the digits that the difference does
@pytest.mark.parametrize("precision,e_lo,tol", [(hpic.HPIC_FP64, 1.1e3, 1e-12), (hpic.HPIC_FP32_MIXED, 5e4, 1e-5)])
@pytest.mark.parametrize("physics", [63, 1 | 2 | 4 | 64, 2 | 64, 1 | 4 | 64])
@pytest.mark.parametrize("n,material", [(20_011, "Au"), (33, "Al")])
def test_energy_range(precision, e_lo, tol, physics, n, material):
    t = W.target(n=(12, 10, 14), material=material)
    run = W.run(seed=5, physics=physics, max_history=2)
    rng = np.random.default_rng(n)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    cells = [rng.integers(1, t[k] - 1, n) + rng.uniform(0.25, 0.75, n) for k in ("nx", "ny", "nz")]
    eps = np.exp(rng.uniform(np.log(e_lo), np.log(1e9), n)) * W.EV / (9.1093837015e-31 * 299792458.0 ** 2)
    u = np.sqrt(eps * (eps + 2))
    d = rng.normal(size=(3, n))
    d /= np.linalg.norm(d, axis=0)
    p = {k: f32(c) * t["dx"] for k, c in zip("xyz", cells)}
    p.update({k: f32(u * v) for k, v in zip(("ux", "uy", "uz"), d)})
    p["tau"] = f32(rng.exponential(0.02, n))
    p["id"] = np.arange(n, dtype=np.uint32)
    laser = W.laser(t, n_macro=0, spot_r=1e-6)
    o = O.OracleSim(t, laser, run)
    g = hpic.Sim(t, laser, run, precision=precision)
    for s in (o, g):
        s.set_particles(p)
        s.set_clock(3, n)
        s.step(1)
    assert_particles_close(by_id(g.particles()), by_id(o.particles()), tol, t["dx"])
    g.close()

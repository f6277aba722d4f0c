"""The batch's tasks are dealt to the blocks in pairs or taken in runs, by the
count of electrons and the block: each electron is pushed once in either order,
as by a single context, with few and many electrons and every shape of block."""
import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

from parity import assert_field_close, assert_particles_close, assert_vector_close

pytestmark = pytest.mark.gpu

SHARES = (0.0, 0.55, 0.07, 0.38)  # of the electrons to each target: one has none


# FP32 without the scatter, whose two branches meet at a rounding; a node's sum
# of up to 5e4 deposits keeps 1e-4 of the largest with each in any order
@pytest.mark.parametrize("precision,blocks", [(hpic.HPIC_FP64, 1), (hpic.HPIC_FP64, 2), (hpic.HPIC_FP32_MIXED, 2),
                                              (hpic.HPIC_FP32_MIXED, 3), (hpic.HPIC_FP32_MIXED, 4),
                                              (hpic.HPIC_FP32_MIXED, 5)])
@pytest.mark.parametrize("total", [37, 5003, 1_700_000])
def test_every_task_once(precision, blocks, total):
    fp32 = precision == hpic.HPIC_FP32_MIXED
    targets = [W.target(n=(20, 18, 23), material=m) for m in ("Au", "Cu", "Al", "Au")]
    counts = [int(total * s) for s in SHARES]
    lasers = [W.laser(t, n_macro=max(c, 1), spot_r=2e-6) for t, c in zip(targets, counts)]
    run = W.run(seed=7, physics=63 & ~2 if fp32 else 63, max_history=2)
    b = hpic.Batch(targets, lasers, run, precision=precision, spare_slots=total)
    b.set_tuning(blocks, 0)
    singles = []
    for t, n in enumerate(counts):
        rng = np.random.default_rng(t)
        s = hpic.Sim(targets[t], lasers[t], dict(run, target_index=t), precision=precision)
        dx = targets[t]["dx"]
        p = {k: rng.uniform(1, targets[t][m] - 1, n) * dx for k, m in zip("xyz", ("nx", "ny", "nz"))}
        p.update({k: rng.normal(size=n) * 5 for k in ("ux", "uy", "uz")})
        p["tau"] = rng.exponential(0.02, n)
        p["id"] = np.arange(n, dtype=np.uint32)
        for x in (s, b.target(t)):
            x.set_particles(p)
            x.set_clock(3000, n)
        s.step(1)
        singles.append(s)
    b.step(1)
    for t, s in enumerate(singles):
        assert_particles_close(b.target(t).particles(), s.particles(), 1e-5 if fp32 else 1e-12, targets[t]["dx"])
        if counts[t]:
            assert_vector_close(b.target(t).grid, s.grid, "j", 1e-4 if fp32 else 1e-11)
            assert_field_close(b.target(t).grid("heat"), s.grid("heat"), 1e-4 if fp32 else 1e-11, "heat")
        assert b.target(t).tallies()["particle_steps"] == counts[t]
        s.close()
    b.close()

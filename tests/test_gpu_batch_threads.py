"""A batch's targets, each used from its own host thread at the same time: what a
thread reads is its own target's grid, and electrons loaded meanwhile stay whole."""
import threading

import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [hpic.HPIC_FP32_MIXED, hpic.HPIC_FP64])
def test_targets_from_their_own_threads(precision):
    sizes = [(18, 20, 22), (18, 20, 22), (20, 18, 16), (7, 9, 8)]
    targets = [W.target(n=n) for n in sizes]
    b = hpic.Batch(targets, None, W.run(seed=1), precision=precision, spare_slots=4096)
    rng = np.random.default_rng(5)
    own = []
    for i, t in enumerate(targets):
        nodes = int(np.prod([m + 1 for m in sizes[i]]))
        for which in ("Ex", "Bz"):
            b.target(i).set_grid(which, (i + 1) * 1e5 + np.arange(nodes))
        p = {k: rng.uniform(0.1, 0.9, 4096) * t[m] * t["dx"] for k, m in zip("xyz", ("nx", "ny", "nz"))}
        p.update({k: rng.normal(size=4096) for k in ("ux", "uy", "uz")})
        p["tau"] = rng.exponential(1.0, 4096)
        p["id"] = np.arange(4096, dtype=np.uint32) + 10000 * i
        b.target(i).set_particles(p)
        own.append((p, {w: b.target(i).grid(w) for w in ("Ex", "Bz")}, b.target(i).particles()))
    wrong, gate = [], threading.Barrier(len(targets))

    def use(i):
        try:
            at_once(i)
        except Exception as e:  # noqa: BLE001
            wrong.append((i, repr(e)))

    def at_once(i):
        p, grids, back = own[i]
        gate.wait()
        for r in range(200):
            for w in ("Ex", "Bz"):
                if not np.array_equal(b.target(i).grid(w), grids[w]):
                    wrong.append((i, r, w))
            b.target(i).set_particles(p)
            got = b.target(i).particles()
            if not all(np.array_equal(got[k], back[k]) for k in back):
                wrong.append((i, r, "electrons"))

    threads = [threading.Thread(target=use, args=(i,)) for i in range(len(targets))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong[:10]
    b.close()

"""The loss-channel estimate at the edges of its split over blocks: a set's
result does not depend on how many others are computed beside it."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def sets(n):
    rng = np.random.default_rng(n)
    return [W.model_point(Z=float(rng.integers(1, 93)), I_Wcm2=10.0 ** rng.uniform(19, 23),
                          L=tuple(10.0 ** rng.uniform(-6, -3, 3)), mechanisms=int(rng.choice([1, 2, 3, 7, 11, 15])))
            for _ in range(n)]


# one set; around a block's 42; around one set per SM; around 42 on each of 152 SMs
@pytest.mark.parametrize("n", [1, 2, 41, 42, 43, 151, 153, 42 * 152, 42 * 152 + 1])
def test_split(n):
    pts = sets(n)
    got = hpic.hpic_model(pts)
    at = sorted({0, n // 3, n // 2, n - 1})
    for i in at:
        alone = hpic.hpic_model([pts[i]])[0]
        assert alone == got[i]
        want = O.model(pts[i])
        for k in hpic.MODEL_E:  # 1e3 steps of RK4, a few roundings of 2^-53 each
            assert abs(got[i][k] - want[k]) <= 1e-11 * want["E_injected"], k

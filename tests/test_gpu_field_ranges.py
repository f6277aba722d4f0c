"""The heating kernel's resistivity over the whole range of temperatures: the
fast expressions hold inside [2^-40, 2^60) K, the general ones outside, and
both must give eta(T) of Eqs. (A4)-(A6) in 64 bits, on the cap's edges too."""
import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def eta_of(t, T):
    kB, me, e, eps0 = 1.380649e-23, 9.1093837015e-31, 1.602176634e-19, 8.8541878128e-12
    kT = kB * T
    hot = 128 * np.pi * eps0 ** 2 / (3 * e ** 4) * np.sqrt(me / (2 * np.pi)) / (t["Zstar"] ** 2 * t["n_i"] * t["lnLambda"]) * kT ** 1.5
    cold = (3 / (4 * np.pi * t["n_i"])) ** (1 / 3) * t["lambda1"] * np.sqrt(me / 3) / np.sqrt(kT)
    return np.minimum(t["lambda2"] * me / (t["Zstar"] * t["n_i"] * e ** 2 * np.maximum(hot, cold)), t["eta_max"])


@pytest.mark.parametrize("precision", [hpic.HPIC_FP32_MIXED, hpic.HPIC_FP64])
@pytest.mark.parametrize("lambda1", [0.0, 7.0])
def test_resistivity_follows_temperature(precision, lambda1):
    t = W.target(n=(13, 6, 7), material="Au", lambda1=lambda1)
    run = W.run(physics=63 | 256, max_history=2)
    n = t["nx"] * t["ny"] * t["nz"]
    band = [T for T in np.logspace(0, 8, 200001) if abs(eta_of(t, T) / t["eta_max"] - 1) < 3e-5]  # the cap's edges
    edges = [2.0 ** -40, np.nextafter(2.0 ** -40, 0), 2.0 ** 60, np.nextafter(2.0 ** 60, 0), 2.0 ** -41, 2.0 ** 61]
    T = np.concatenate([edges, band[:100], np.logspace(-14, 19, n)])[:n]
    s = hpic.Sim(t, None, run, precision=precision)
    s.set_grid("T", T)
    s.set_grid("Ti", T * (1 - 1e-6))  # the exchange touches every cell
    s.step(1)
    T1, eta = s.grid("T"), s.grid("eta")
    # a few roundings of T^1.5 and of the constants, each 2^-53
    assert np.max(np.abs(eta / eta_of(t, T1) - 1)) < 1e-14
    assert np.all(eta <= t["eta_max"])
    s.close()

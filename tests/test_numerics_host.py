"""The push's own FP64 functions, built for the host with the hardware's estimates at
their worst, against 60-digit values: each within the error that the library function
it stands for is given, over the range that the push uses.

Unit of the errors: the last place (ulp) of the exact result.  log of CUDA's library is
given 1, sincospi 2, sqrt and division are rounded (1/2)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
mp.mp.dps = 60

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2107_01723_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("numerics") / "numerics.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    "-o", so, os.path.join(HERE, "numerics_host.cpp")], check=True)
    return C.CDLL(so)


def call(fn, *arrays, outs=1):
    n = len(arrays[0])
    out = [np.empty(n) for _ in range(outs)]
    fn(*[a.ctypes.data_as(C.c_void_p) for a in (*arrays, *out)], C.c_long(n))
    return out[0] if outs == 1 else out


def worst(got, exact, given):
    """The largest error in ulp of the exact result, and where."""
    e = [abs(mp.mpf(float(g)) - x) / mp.mpf(float(np.spacing(abs(float(x))))) for g, x in zip(got, exact)]
    i = int(np.argmax([float(v) for v in e]))
    return float(e[i]), given[i]


def deviates(m):
    return (np.asarray(m, np.uint64) << 9).astype(np.uint32)


def test_log_of_a_deviate(lib):
    """ln u of the 23-bit deviate, also just below 1, where it is small."""
    rng = np.random.default_rng(1)
    top = (1 << 23) - 1
    m = np.unique(np.concatenate([np.arange(64), top - np.arange(64), top - (np.logspace(0, 6.8, 600)).astype(int),
                                  rng.integers(0, top, 1500)]))
    x = (m + 0.5) * 2.0**-23
    e, at = worst(call(lib.run_log, x), [mp.log(mp.mpf(v)) for v in x], x)
    assert e <= 1.0, (e, at)


def test_log_of_any_number(lib):
    rng = np.random.default_rng(2)
    near = np.concatenate([1 + s * np.logspace(-15, -0.5, 400) for s in (1, -1)])
    rows = (1 + (np.arange(512) + 0.5) / 512)  # the rows' ends
    x = np.concatenate([near, rows, np.nextafter(rows, 0), 2.0**rng.uniform(-1000, 1000, 600),
                        2.0**rng.uniform(-40, 40, 1500), [2.0**-1022, np.finfo(float).max, 1.0]])
    exact = [mp.log(mp.mpf(v)) for v in x]
    keep = [i for i, v in enumerate(exact) if v != 0]
    got = call(lib.run_log, x)
    assert got[x == 1.0] == 0
    e, at = worst(got[keep], [exact[i] for i in keep], x[keep])
    assert e <= 1.05, (e, at)  # 1/2 for the result, 1/2 for r in the rows next to 1


def test_log_for_fp32_results(lib):
    """In two parts, to 2^-33: of a temperature, and next to 1 and to the rows' ends."""
    rng = np.random.default_rng(6)
    rows = (1 + (np.arange(512) + 0.5) / 512)
    x = np.concatenate([2.0**rng.uniform(-40, 60, 3000), rows, np.nextafter(rows, 0), np.nextafter(rows, 3),
                        1 + np.logspace(-15, -1, 100), 1 - np.logspace(-15, -1, 100)])
    base, rest = call(lib.run_log_parts, x, outs=2)
    e = [float(abs(mp.mpf(float(b)) + mp.mpf(float(r)) - mp.log(mp.mpf(float(v))))) for b, r, v in zip(base, rest, x)]
    assert max(e) <= 2.0**-33, (max(e) * 2.0**33, x[int(np.argmax(e))])


def test_circle(lib):
    """Sine and cosine of the deviate, also at the quarters, where one is small."""
    rng = np.random.default_rng(3)
    quarters = np.concatenate([q * (1 << 21) + np.concatenate([np.arange(-40, 40), s * np.logspace(0.1, 6, 150).astype(int)])
                               for q in range(4) for s in (1, -1)])
    m = np.unique(np.concatenate([quarters % (1 << 23), rng.integers(0, 1 << 23, 1500)]))
    turn = [(mp.mpf(int(v)) + mp.mpf(1) / 2) / 2**23 for v in m]
    s, c = call(lib.run_turn, deviates(m), outs=2)
    for got, exact in ((s, [mp.sin(2 * mp.pi * t) for t in turn]), (c, [mp.cos(2 * mp.pi * t) for t in turn])):
        e, at = worst(got, exact, m)
        assert e <= 2.0, (e, at)


@pytest.mark.parametrize("off", [-2, 0, 2])
def test_quotients_and_roots(lib, off):
    """Rounded but for rare last places: 1/2 and what three terms of the residual's
    series leave at an estimate of two last places off (4e-7 cubed: below 1e-3)."""
    rng = np.random.default_rng(4)
    x = np.concatenate([2.0**rng.uniform(-30, 30, 1500), 1 + rng.uniform(0, 1e-6, 300), 1 + 2.0**rng.uniform(-40, 2, 300)])
    y = np.concatenate([2.0**rng.uniform(-30, 30, 1800), rng.uniform(1, 2, 300)])
    lib.set_off(off)
    try:
        X, Y = [mp.mpf(v) for v in x], [mp.mpf(v) for v in y]
        for fn, given, exact in ((lib.run_rcp, (x,), [1 / v for v in X]),
                                 (lib.run_rsqrt, (x,), [1 / mp.sqrt(v) for v in X]),
                                 (lib.run_sqrt, (x,), [mp.sqrt(v) for v in X]),
                                 (lib.run_div, (y, x), [b / a for a, b in zip(X, Y)])):
            e, at = worst(call(fn, *given), exact, x)
            assert e <= 0.501, (e, at)
    finally:
        lib.set_off(0)


@pytest.mark.parametrize("steps", [1, 3, 40])
@pytest.mark.parametrize("kind", ["alike", "spread", "signs"])
def test_warp_sums(lib, steps, kind):
    """FP32 values summed by a warp as exactly as an FP64 sum of them: within one
    rounding in FP64 of the exact sum, and of what the values' own size allows."""
    import math
    lib.warp_total.restype = C.c_double
    rng = np.random.default_rng(steps)
    for _ in range(200):
        x = rng.uniform(0.5, 1, 32 * steps)
        if kind != "alike":
            x *= 2.0**rng.uniform(-24, 0, x.size)
        if kind == "signs":
            x *= rng.choice([-1, 1], x.size)
        x = x.astype(np.float32)
        exact = math.fsum(x.astype(float))
        got = lib.warp_total(x.ctypes.data_as(C.c_void_p), C.c_long(steps))
        # the result's rounding, and below that the last part's (24 bits, 48 below the largest)
        bound = 2.0**-53 * abs(exact) + 2.0**-68 * float(np.sum(np.abs(x, dtype=float)))
        assert abs(got - exact) <= bound, (got, exact, abs(got - exact) / bound)
    inf = np.zeros(32, np.float32)
    inf[3] = np.inf
    assert lib.warp_total(inf.ctypes.data_as(C.c_void_p), C.c_long(1)) == np.inf


def test_rotation(lib):
    """Against the frame's vectors summed out in long doubles, on both hemispheres, at
    the poles and at the equator: some ten roundings of numbers below 2."""
    L = np.longdouble
    rng = np.random.default_rng(8)
    n = 4000
    d = rng.normal(size=(n, 3))
    d[:200, :2] *= 1e-9
    d[200:400, 2] *= 1e-17
    d /= np.linalg.norm(d, axis=1)[:, None]
    d[:4] = [[0, 0, 1], [0, 0, -1], [1, 0, 0], [0, 1, -0.0]]
    theta, phi = rng.normal(size=n) * 0.3, rng.uniform(0, 2 * np.pi, n)
    ct, st, cp, sp = np.cos(theta), np.sin(theta), np.cos(phi), np.sin(phi)
    x, y, z = d.T.astype(L)
    sg = np.where(z >= 0, L(1), L(-1))
    a = -1 / (sg + z)
    b = x * y * a
    e1 = np.stack([1 + sg * x * x * a, sg * b, -sg * x])
    e2 = np.stack([b, sg + y * y * a, -y])
    want = d.T.astype(L) * ct + (e1 * cp + e2 * sp) * st.astype(L)
    got = np.ascontiguousarray(d)
    lib.run_rotate(*[v.ctypes.data_as(C.c_void_p) for v in (got, ct, st, cp, sp)], C.c_long(n))
    assert float(np.max(np.abs(got.T - want))) <= 10 * 2.0**-52

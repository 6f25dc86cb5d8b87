"""The integer-weight WENO5 reconstruction (csrc/janc_weno.cuh) on the CPU
against exact rational arithmetic: face values, derivatives, the reciprocal
and the conversion, over smooth, discontinuous, tiny, huge and mixed windows."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction as Q

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    out = str(tmp_path_factory.mktemp("wh") / "libweno_harness.so")
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-shared", "-fPIC",
                    os.path.join(HERE, "weno_harness.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _faces(lib, Fp, Fm, eps):
    n, ln = Fp.shape
    s, d = np.zeros(n), np.zeros((n, 8))
    lib.wh_faces(n, ln - 6, _ptr(Fp), _ptr(Fm), ctypes.c_double(eps), _ptr(s), _ptr(d))
    return s, d


def _exact(f, eps):
    """WENO5-JS value at the right face of f[2] and its derivative with
    respect to the four differences, in rationals."""
    D = [f[k + 1] - f[k] for k in range(4)]
    C = [4 * D[0] ** 2 - 11 * D[0] * D[1] + 10 * D[1] ** 2, 4 * D[1] ** 2 - 5 * D[1] * D[2] + 4 * D[2] ** 2,
         10 * D[2] ** 2 - 11 * D[2] * D[3] + 4 * D[3] ** 2]
    C = [c + 3 * eps for c in C]
    dC = [[8 * D[0] - 11 * D[1], 20 * D[1] - 11 * D[0], 0, 0], [0, 8 * D[1] - 5 * D[2], 8 * D[2] - 5 * D[1], 0],
          [0, 0, 20 * D[2] - 11 * D[3], 8 * D[3] - 11 * D[2]]]
    a = [Q(g) / c ** 2 for g, c in zip((1, 6, 3), C)]
    s = sum(a)
    w = [x / s for x in a]
    q = [(5 * D[1] - 2 * D[0]) / 6, (D[1] + 2 * D[2]) / 6, (4 * D[2] - D[3]) / 6]
    dq = [[Q(-2, 6), Q(5, 6), 0, 0], [0, Q(1, 6), Q(2, 6), 0], [0, 0, Q(4, 6), Q(-1, 6)]]
    r = sum(x * y for x, y in zip(w, q))
    g = [sum(w[k] * dq[k][m] - 2 * w[k] * (q[k] - r) * dC[k][m] / C[k] for k in range(3)) for m in range(4)]
    return f[2] + r, g


def _windows(kind, n, ln, rng):
    x = rng.uniform(0, 6.28, (n, 1)) + rng.uniform(0, 0.4, (n, 1)) * np.arange(ln)
    jump = np.arange(ln)[None] >= rng.integers(1, ln, (n, 1))
    return {
        "smooth": 1e5 * (2 + np.sin(x)),
        "shock": 1e5 * (1 + 0.1 * np.sin(x)) + jump * rng.uniform(0, 3e6, (n, 1)),
        "energy_shock": 1e9 * (1 + 1e-3 * rng.uniform(size=(n, ln)) + 10 * jump),
        "noise": rng.standard_normal((n, ln)),
        "below_eps": 1e-8 * rng.standard_normal((n, ln)),
        "around_eps": 1e-3 * (2 + np.sin(3 * x)),
        "half_zero": np.where(jump, 0.0, 1e5 * (1 + 0.01 * rng.uniform(size=(n, ln)))),
        "mixed": rng.standard_normal((n, ln)) * np.exp(12 * rng.standard_normal((n, ln))),
        "tie": rng.integers(-3, 4, (n, ln)).astype(float),
        "huge": 1e80 * rng.standard_normal((n, ln)),
        "uniform": np.broadcast_to(rng.standard_normal((n, 1)), (n, ln)),
    }[kind].astype(np.float64)


KINDS = ("smooth", "shock", "energy_shock", "noise", "below_eps", "around_eps", "half_zero", "mixed", "tie", "huge", "uniform")


@pytest.mark.parametrize("slide", [0, 5])
@pytest.mark.parametrize("kind", KINDS)
def test_faces_and_derivatives(lib, kind, slide):
    rng = np.random.default_rng([KINDS.index(kind), slide])
    n, ln, eps = 150, 6 + slide, 1e-6
    Fp = np.ascontiguousarray(_windows(kind, n, ln, rng))
    Fm = np.ascontiguousarray(_windows(kind, n, ln, rng))
    s, d = _faces(lib, Fp, Fm, eps)
    for i in range(n):
        p, m = [Q(float(v)) for v in Fp[i, slide:]], [Q(float(v)) for v in Fm[i, slide:]]
        vp, gp = _exact(p[0:5], Q(eps))
        vm, gm = _exact(m[5:0:-1], Q(eps))
        # 10 roundings, each at most half an ulp of a partial sum bounded by the largest value
        # (centre values) or twice the largest difference (the small terms)
        scale = max(abs(v) for v in p + m)
        assert abs(Q(s[i]) - (vp + vm)) <= 12 * Q(2) ** -53 * scale
        # the mirrored window's differences run backwards with the sign changed: D4..D1
        gm = [-g for g in gm[::-1]]
        # second derivative terms: |g| <= 8, every factor good to a few ulps of the largest difference,
        # whose square the forms are at least 0.7 of
        for a, b in zip(d[i], gp + gm):
            assert abs(Q(float(a)) - b) <= Q(2) ** -44 * max(1, abs(b))
    if kind == "uniform":
        assert np.array_equal(s, Fp[:, 0] + Fm[:, 0])


def test_nonfinite_values_stay_nonfinite(lib):
    F = np.ones((12, 6))
    F[np.arange(6), np.arange(6)] = np.inf
    F[6 + np.arange(6), np.arange(6)] = np.nan
    s, _ = _faces(lib, F, F, 1e-6)
    assert not np.isfinite(s).any()


def test_reciprocal_and_conversion(lib):
    rng = np.random.default_rng(3)
    x = [2 ** 56, 2 ** 56 + 1, 2 ** 63, 2 ** 63 + 1, 2 ** 64 - 1, 2 ** 64 - 2 ** 32, 2 ** 57 - 1, 3 * 2 ** 61]
    x += [int(v) | 2 ** 56 for v in rng.integers(0, 2 ** 63, 20000, dtype=np.uint64) >> rng.integers(0, 7, 20000).astype(np.uint64)]
    x = np.array(x, dtype=np.uint64)
    n = x.size
    y, z, b = np.zeros(n, np.uint64), np.zeros(n, np.int32), np.zeros(n)
    lib.wh_soft(n, _ptr(x), _ptr(y), _ptr(z), _ptr(b))
    for xi, yi, zi, bi in zip(x.tolist(), y.tolist(), z.tolist(), b.tolist()):
        assert zi == 64 - xi.bit_length()
        assert abs(Q(yi) - Q(2 ** 127, xi << zi)) <= 8
        assert 0 <= Q(xi, 2 ** 64) - Q(bi) < Q(xi, 2 ** 64) * Q(2) ** -52


def _functions(lib, x):
    x = np.ascontiguousarray(x, dtype=np.float64)
    out = [np.zeros(x.size) for _ in range(3)]
    lib.wh_functions(x.size, _ptr(x), *[_ptr(o) for o in out])
    return out


def test_exponential_logarithm_reciprocal(lib):
    """exp within 0.9 units in the last place (half an ulp of rounding, the
    argument cut at 2^-54, the power of two good to 2^-57), ln within 2^-53
    absolute plus half an ulp, 1/x within 0.51."""
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 160
    rng = np.random.default_rng(5)
    x = np.concatenate([rng.uniform(-707.9, 707.9, 3000), rng.uniform(-40, 40, 3000), rng.normal(0, 1e-3, 500),
                        [0.0, -0.0, 1e-300, -1e-300, 5e-324, 1.0, -1.0, 512.0, -512.0, 511.99999, np.log(2.0)]])
    e, _, _ = _functions(lib, x)
    for xi, ei in zip(x, e):
        assert abs(mp.mpf(float(ei)) - mp.exp(mp.mpf(float(xi)))) <= 0.9 * np.spacing(ei)
    t = np.concatenate([rng.uniform(2, 1e4, 4000), 10.0 ** rng.uniform(0.31, 300, 1000), 2.0 ** np.arange(1, 1000, 37),
                        np.nextafter(2.0 ** np.arange(2, 1000, 37), 0.0)])
    _, l, _ = _functions(lib, t)
    for ti, li in zip(t, l):
        assert abs(mp.mpf(float(li)) - mp.log(mp.mpf(float(ti)))) <= 0.5 * np.spacing(li) + 2.0 ** -53 * max(1.0, li / 512)
    y = 10.0 ** rng.uniform(-300, 300, 4000) * rng.choice([-1.0, 1.0], 4000) * rng.uniform(1, 2, 4000)
    y = np.concatenate([y, 2.0 ** np.arange(-1000, 1000, 41), np.nextafter(2.0 ** np.arange(-1000, 1000, 41), 0.0)])
    _, _, r = _functions(lib, y)
    for yi, ri in zip(y, r):
        assert abs(Q(float(ri)) - 1 / Q(float(yi))) <= Q(51, 100) * Q(float(np.spacing(abs(ri))))
    _, _, r = _functions(lib, np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-310, 8e307]))
    assert np.isnan(r[:6]).all() and r[6] == 0.0


def test_square_root_and_signed_conversion(lib):
    rng = np.random.default_rng(6)
    d = rng.integers(2 ** 62, 2 ** 64, 20000, dtype=np.uint64, endpoint=False)
    d = np.concatenate([d, np.array([2 ** 62, 2 ** 62 + 1, 2 ** 63, 2 ** 64 - 1, 2 ** 63 - 1], dtype=np.uint64)])
    s = np.zeros(d.size, np.uint64)
    lib.wh_sqrt(d.size, _ptr(d), _ptr(s))
    for di, si in zip(d.tolist(), s.tolist()):
        # within 16 units: s^2 against d 2^64
        assert (si - 16) ** 2 <= di << 64 <= (si + 16) ** 2
    a = rng.integers(-2 ** 62, 2 ** 62, 5000) >> rng.integers(0, 62, 5000)
    a = np.concatenate([a, [0, 1, -1, 2 ** 31, 2 ** 32, -2 ** 32, 2 ** 62, -2 ** 62, 2 ** 32 - 1]])
    for e in (0, -1000, 900):
        x = np.zeros(a.size)
        lib.wh_signed(a.size, _ptr(a), e, _ptr(x))
        for ai, xi in zip(a.tolist(), x.tolist()):
            want = Q(ai) * Q(2) ** e
            assert abs(Q(xi) - want) <= Q(float(np.spacing(abs(xi)))) / 2


def test_scaled_conversion_fixed_exponential_and_floats(lib):
    """a 2^e rounded to nearest and 0 below the normal range; 2^(a 2^-54) within
    0.9 units in the last place as exp; floats cut towards zero."""
    rng = np.random.default_rng(8)
    a = rng.integers(-2 ** 63 + 1, 2 ** 63 - 1, 4000) >> rng.integers(0, 63, 4000)
    a = np.concatenate([a, [0, 1, -1, 2 ** 31, 2 ** 32 - 1, 2 ** 32, -2 ** 62, 2 ** 63 - 1]])
    x = np.zeros(a.size)
    for e in (0, -1022, -1060, -1085, -1200, 900):
        lib.wh_scaled(a.size, _ptr(a), e, _ptr(x))
        for ai, xi in zip(a.tolist(), x.tolist()):
            want = Q(ai) * Q(2) ** e
            if abs(want) < Q(2) ** -1022:
                assert xi == 0.0 or abs(xi) == 2.0 ** -1022
            else:
                assert abs(Q(xi) - want) <= Q(float(np.spacing(abs(xi)))) / 2
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 160
    k = np.concatenate([rng.integers(-2 ** 63, 2 ** 63 - 1, 3000), rng.integers(-2 ** 54, 2 ** 54, 1000),
                        np.array([0, 1, -1, 2 ** 54, -2 ** 54, 2 ** 54 - 1, 510 * 2 ** 54, -512 * 2 ** 54])])
    y = np.zeros(k.size)
    lib.wh_exp2(k.size, _ptr(k), _ptr(y))
    for ki, yi in zip(k.tolist(), y.tolist()):
        assert abs(mp.mpf(yi) - mp.mpf(2) ** (mp.mpf(ki) / 2 ** 54)) <= 0.9 * np.spacing(yi)
    f = np.concatenate([rng.standard_normal(2000) * 10.0 ** rng.uniform(-36, 36, 2000), [1.0, -1.0, 2.0 ** -126, -3.0e38]])
    g = np.zeros(f.size)
    lib.wh_float(f.size, _ptr(f), _ptr(g))
    assert np.all(np.abs(g) <= np.abs(f)) and np.all(np.abs(f - g) < 2.0 ** -23 * np.abs(f)) and np.all(f * g > 0)
    z = np.array([0.0, -0.0, 1e-39, 5e-324])
    lib.wh_float(4, _ptr(z), _ptr(g))
    assert np.all(np.abs(g[:4]) <= 2.0 ** -127)


@pytest.mark.parametrize("eps", [1e-130, 1e-140, 1e-150, 1e-200, 1e-300])
def test_derivatives_at_small_epsilon(lib, eps):
    """Indicators up to 2^2050 apart, where a weight leaves the range of doubles:
    one, two or three values of a window equal (a flat substencil) beside
    differences of 1e-3 to 1e10. The bars of test_faces_and_derivatives."""
    rng = np.random.default_rng(int(-np.log10(eps)))
    n = 120
    jump = np.arange(6)[None] >= rng.integers(0, 7, (n, 1))
    size = 10.0 ** rng.uniform(-3, 10, (n, 6))
    for F in (jump * size[:, :1], np.where(jump, size, 1e9), size * rng.standard_normal((n, 6))):
        F = np.ascontiguousarray(F)
        s, d = _faces(lib, F, F, eps)
        for i in range(n):
            f = [Q(float(v)) for v in F[i]]
            vp, gp = _exact(f[0:5], Q(eps))
            vm, gm = _exact(f[5:0:-1], Q(eps))
            assert abs(Q(s[i]) - (vp + vm)) <= 12 * Q(2) ** -53 * max(abs(v) for v in f)
            for a, b in zip(d[i], gp + [-g for g in gm[::-1]]):
                assert np.isfinite(a) and abs(Q(float(a)) - b) <= Q(2) ** -44 * max(1, abs(b))

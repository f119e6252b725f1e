"""Host checks of the integer arithmetic of fx.cuh, compiled with the host
compiler: each function against exact rationals or 60-digit decimals over its
range and at its ends."""

import ctypes
import subprocess
from decimal import Decimal, localcontext
from fractions import Fraction
from pathlib import Path

import numpy as np
import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_1712_00953_gb300" / "csrc"
SRC = """
#include "fx.cuh"
using namespace rk;
static const uint64_t tab[] = {RK_FX_EXP2_VALUES};
static const uint64_t ic[] = {RK_FX_INV_C_VALUES}, lc[] = {RK_FX_LOG2_C_VALUES};
extern "C" {
double t_exp(double x) { return fx::exp_double(x, tab); }
uint64_t t_log2(double x) { return fx::log2_fixed(x, ic, lc); }
uint64_t t_rcp(double T, double r) { return fx::recip_fixed70(T, r); }
double t_scale(double x, double D) {  // e^x D as the reactions form it
  const uint64_t L = fx::log2e_fixed(x);
  return fx::mul_sig(fx::exp2_sig(L, tab), fx::exponent(L), D);
}
double t_sum(const double* v, int n, int hb) {  // sum of v[i], every other one subtracted
  int em = 0;
  for (int i = 0; i < n; ++i) { int e = (fx::hi32(v[i]) >> 20) & 0x7ff; if (e > em) em = e; }
  fx::Wide a = {0, 0};
  for (int i = 0; i < n; ++i) {
    const fx::Wide w = fx::to_grid(v[i], em, hb);
    if (i & 1) fx::sub(a, w.hi, w.lo); else fx::add(a, w.hi, w.lo);
  }
  return fx::from_grid(a, em, hb);
}
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", str(CSRC), str(d / "t.cpp"), "-o",
                    str(d / "t.so")], check=True)
    lib = ctypes.CDLL(str(d / "t.so"))
    D, U = ctypes.c_double, ctypes.c_uint64
    for name, res, args in (("t_exp", D, [D]), ("t_log2", U, [D]), ("t_rcp", U, [D, D]), ("t_scale", D, [D, D]),
                            ("t_sum", D, [ctypes.c_void_p, ctypes.c_int, ctypes.c_int])):
        f = getattr(lib, name)
        f.restype, f.argtypes = res, args
    return lib


def test_header_is_the_generator_output(capsys):
    import importlib.util

    spec = importlib.util.spec_from_file_location("gen_fx_table", CSRC / "gen_fx_table.py")
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    mod.main()
    assert capsys.readouterr().out.strip() == (CSRC / "fx_table.h").read_text().strip()


def test_exp_within_an_ulp_and_a_quarter(fx):
    """|x| < 708: the argument's product is cut at 2^-53 for the largest |x| (1 unit
    = 0.7 ulp at worst) and the result rounded once (0.5 ulp)."""
    rng = np.random.default_rng(1)
    xs = np.concatenate([rng.uniform(-707.9, 707.9, 1500), rng.uniform(-3, 3, 500),
                         10.0 ** rng.uniform(-300, 0, 100), [0.0, -0.0, 707.99, -707.99, 1e-17, -1e-17, 0.5, -0.5]])
    with localcontext() as c:
        c.prec = 50
        for x in xs:
            y, e = fx.t_exp(float(x)), Decimal(float(x)).exp()
            assert abs(Decimal(y) - e) <= Decimal("1.25") * Decimal(float(np.spacing(float(e)))), x


def test_log2_and_reciprocal_of_temperatures(fx):
    """T in [150, 16000): log2 T to 2^-54 absolute (its coefficients' truncation is
    four units of 2^-56), 2^70 / T to 2 units from a reciprocal one ulp off either way."""
    rng = np.random.default_rng(2)
    Ts = np.concatenate([rng.uniform(150.0, 16000.0, 1500), 2.0 ** np.arange(8, 14), [150.0, 15999.999],
                         np.nextafter(2.0 ** np.arange(8, 14), 0), np.nextafter(2.0 ** np.arange(8, 14), 1e9)])
    with localcontext() as c:
        c.prec = 50
        ln2 = Decimal(2).ln()
        for T in Ts:
            T = float(T)
            lg = Decimal(T).ln() / ln2
            assert abs(Decimal(fx.t_log2(T)) / Decimal(2) ** 59 - lg) < Decimal(2) ** -54, T
            for r in (1.0 / T, float(np.nextafter(1.0 / T, 0)), float(np.nextafter(1.0 / T, 1))):
                assert abs(Fraction(fx.t_rcp(T, r)) - Fraction(2) ** 70 / Fraction(T)) <= 2, (T, r)


def test_scaled_product(fx):
    """e^x D: 2^-52 of the fixed-point argument (1.1 units: 1.6 ulp) and two roundings;
    zero, infinite, NaN and out-of-range products."""
    rng = np.random.default_rng(3)
    with localcontext() as c:
        c.prec = 50
        for x, D in zip(rng.uniform(-300, 300, 800), (rng.random(800) - 0.5) * 10.0 ** rng.uniform(-100, 100, 800)):
            y, e = fx.t_scale(float(x), float(D)), Decimal(float(x)).exp() * Decimal(float(D))
            assert abs(Decimal(y) - e) <= Decimal("2.5") * Decimal(float(np.spacing(abs(float(e))))), (x, D)
    assert fx.t_scale(5.0, 0.0) == 0.0 and fx.t_scale(-600.0, 1e-200) == 0.0
    assert fx.t_scale(600.0, 1e200) == np.inf and fx.t_scale(600.0, -1e200) == -np.inf
    assert fx.t_scale(-1.0, np.inf) == np.inf and np.isnan(fx.t_scale(1.0, np.nan))


@pytest.mark.parametrize("spread", [0, 30, 60, 200])
def test_grid_sums_are_exact(fx, spread):
    """Sums of values over `spread` binary orders of magnitude, cancelling ones among
    them: the exact sum of what lies above 2^-(126 - hb) of the largest, rounded once."""
    rng = np.random.default_rng(4 + spread)
    hb = 8
    for n in (1, 2, 3, 40, 120):
        for _ in range(40):
            v = (rng.random(n) - 0.5) * 2.0 ** rng.uniform(-spread, 0, n) * 2.0 ** rng.integers(-100, 100)
            if n > 3:
                v[1], v[3] = v[0], v[0] * (1 + 2.0 ** -52)
                v[2] = v[0]
            v = np.ascontiguousarray(v)
            exact = sum((Fraction(float(x)) * (-1 if i & 1 else 1) for i, x in enumerate(v)), Fraction(0))
            got = Fraction(fx.t_sum(v.ctypes.data, n, hb))
            cut = n * Fraction(float(np.max(np.abs(v)))) / Fraction(2) ** (126 - hb - 2)
            half = Fraction(float(np.spacing(abs(float(exact))))) / 2
            assert abs(got - exact) <= half * (1 + Fraction(1, 2 ** 10)) + cut, (n, v)
    z = np.zeros(4)
    assert fx.t_sum(z.ctypes.data, 4, hb) == 0.0


def test_scaled_product_below_the_normal_range(fx):
    """Subnormal factors and results: the same relative error where the result is normal
    (test_scaled_product), else within one unit in its last place, the smallest double."""
    rng = np.random.default_rng(5)
    xs, Ds = rng.uniform(-700, 300, 1500), (rng.random(1500) - 0.5) * 10.0 ** rng.uniform(-323, -100, 1500)
    xs[:4], Ds[:4] = [0.0, -0.5, 700.0, -3.0], [5e-324, 5e-324, 5e-324, 2.2250738585072014e-308]
    subnormal = 0
    with localcontext() as c:
        c.prec, c.Emin = 50, -2000
        for x, D in zip(xs, Ds):
            y, e = fx.t_scale(float(x), float(D)), Decimal(float(x)).exp() * Decimal(float(D))
            place = Decimal(float(np.spacing(abs(float(e)))))
            subnormal += 0 < abs(y) < 2.3e-308
            assert abs(Decimal(y) - e) <= (Decimal("2.5") if abs(float(e)) >= 2.3e-308 else 1) * place, (x, D)
    assert subnormal > 30
    assert fx.t_scale(-700.0, -1e-300) == 0.0

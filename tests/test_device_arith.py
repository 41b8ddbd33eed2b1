"""CPU checks of arithmetic identities the CUDA kernels rely on for bit-exact
agreement with the oracle (no GPU needed; exact rational arithmetic stands in
for the FP64 units).

Division by a constant c in {3, 12, 20} (the predictor's dt/3 and the
corrector's a2/12, a3/20, a2/3): the kernels form q0 = RN(a y) with
y = RN(1/c), the exact residual r = a - c q0 (one FMA) and q = RN(q0 + r y)
(one FMA), which is RN(a / c) by Markstein's theorem (IBM J. Res. Dev. 34,
1990: q0 within one ulp of a/c, y within half an ulp of 1/c).  Here the three
steps are replayed exactly and compared with the correctly rounded quotient
on random operands over a wide exponent range and on operands whose quotient
lies next to a rounding midpoint.

Subtraction as the addition of the negated operand (the packed two-lane adds
of the DS force kernels): RN(a + (-b)) = RN(a - b) bit for bit in float32,
signed zeros, subnormals, infinities and NaN included.
"""
import math
import random
from fractions import Fraction as F

import pytest

CONSTS = (3, 12, 20)


def _markstein(a, c):
    y = 1.0 / c                       # RN(1/c), as the compiler folds it
    q0 = float(F(a) * F(y))           # RN(a * y)
    r = F(a) - F(q0) * c              # a - c q0, which the FMA forms exactly
    assert float(r) == r, "residual not representable"
    return float(F(q0) + r * F(y))    # RN(q0 + r y), the second FMA


def _operands(rng, count):
    for _ in range(count):
        m = rng.getrandbits(52) | (1 << 52)
        e = rng.randint(-200, 200)
        yield math.ldexp(m, e - 52) * rng.choice((1.0, -1.0))


@pytest.mark.parametrize("c", CONSTS)
def test_division_by_constant_is_correctly_rounded(c):
    rng = random.Random(c)
    for a in _operands(rng, 20000):
        assert _markstein(a, c) == float(F(a) / c), (a, c)


@pytest.mark.parametrize("c", CONSTS)
def test_division_by_constant_near_midpoints(c):
    # quotients within a few ulps of a midpoint between two doubles
    rng = random.Random(100 + c)
    for _ in range(4000):
        k = rng.getrandbits(52) | (1 << 52)
        mid = F(2 * k + 1, 2) * F(2) ** rng.randint(-60, 60)
        a0 = float(mid * c)
        for d in range(-3, 4):
            a = a0
            for _ in range(abs(d)):
                a = math.nextafter(a, math.inf if d > 0 else -math.inf)
            assert _markstein(a, c) == float(F(a) / c), (a, c)


def test_fast_path_limits_cover_the_faithful_quotient():
    # the kernels take the three-step path only for 2^-900 < |a| < 2^1000;
    # there neither a y nor the residual leaves the normal range
    for c in CONSTS:
        for a in (math.ldexp(1.0, -899), math.ldexp(1.999, 999), -math.ldexp(1.5, -899)):
            assert _markstein(a, c) == float(F(a) / c)


def test_adding_the_negation_rounds_as_the_subtraction():
    # The DS force kernels take the x and y components of x_j - x_i (hi and
    # lo parts) and of v_j - v_i as packed two-lane adds of the negated i
    # values: RN(a + (-b)) must be RN(a - b) bit for bit, signed zeros
    # included, for the forces to equal the scalar form's.  Negation is exact
    # in IEEE arithmetic, so the two are one operation; checked here in float32
    # on random magnitudes over the whole range, on equal and nearly equal
    # operands, and on the special values.
    np = pytest.importorskip("numpy")
    rng = np.random.default_rng(17)
    k = 200000
    mant = rng.uniform(-2.0, 2.0, size=(2, k))
    expo = rng.integers(-140, 128, size=(2, k))
    with np.errstate(over="ignore"):
        ab = np.ldexp(mant, expo).astype(np.float32)   # subnormal to overflowing
    a, b = ab[0], ab[1]
    b2 = np.nextafter(a, np.float32(np.inf))            # one ulp apart
    special = np.array([0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, np.nan, 1e-45, -1e-45,
                        np.finfo(np.float32).max, -np.finfo(np.float32).max,
                        np.finfo(np.float32).tiny], dtype=np.float32)
    sa, sb = np.meshgrid(special, special)
    with np.errstate(over="ignore", invalid="ignore"):
        for x, y in ((a, b), (a, a), (a, b2), (b2, a), (sa.ravel(), sb.ravel())):
            x = np.asarray(x, dtype=np.float32)
            y = np.asarray(y, dtype=np.float32)
            sub = x - y
            add = x + (-y)
            assert sub.dtype == np.float32 and add.dtype == np.float32
            same = (sub.view(np.uint32) == add.view(np.uint32)) | (np.isnan(sub) & np.isnan(add))
            assert same.all(), (x[~same][:5], y[~same][:5])


np = pytest.importorskip("numpy")


def _split_int(x):
    # split_ds_int of nb_device.cuh in numpy integers: RN32(x), RN32(x - RN32(x))
    b = x.view(np.uint64)
    xh, xl = (b >> np.uint64(32)).astype(np.int64), (b & np.uint64(0xffffffff)).astype(np.int64)
    e = (xh >> 20) & 0x7ff
    t = ((((xh & 0x7fffffff) - (896 << 20)) << 3) & 0xffffffff) | (xl >> 29)
    r = xl & 0x1fffffff
    up = (r + (t & 1) > 0x10000000).astype(np.int64)
    hi = ((t + up) | (xh & 0x80000000)).astype(np.uint32).view(np.float32)
    r = r - up * 0x20000000
    r = np.where(xh & 0x80000000, -r, r)
    lo = r.astype(np.float32) * ((e - (1075 - 127)) << 23).astype(np.uint32).view(np.float32)
    return hi, lo


def test_integer_split_into_double_single():
    # random values over the exponents that take the integer form, ties and
    # near-ties of both roundings, and carries into the next binade
    rng = np.random.RandomState(11)
    e = rng.randint(1023 - 70, 1023 + 119, 200000).astype(np.uint64)
    m = rng.randint(0, 1 << 52, 200000, dtype=np.int64).astype(np.uint64)
    m[:20000] = (m[:20000] & ~np.uint64(0x1fffffff)) | np.uint64(0x10000000)
    m[20000:40000] = (m[20000:40000] & ~np.uint64(0x1fffffff)) + rng.randint(0x0fffffff, 0x10000002, 20000).astype(np.uint64)
    m[40000:41000] = np.uint64((1 << 52) - 1) - rng.randint(0, 1 << 30, 1000).astype(np.uint64)
    m[41000:42000] = 0
    s = rng.randint(0, 2, 200000).astype(np.uint64)
    x = ((s << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)
    hi, lo = _split_int(x)
    want = x.astype(np.float32)
    assert np.array_equal(hi.view(np.uint32), want.view(np.uint32))
    rest = (x - want.astype(np.float64)).astype(np.float32)
    assert np.array_equal(lo.view(np.uint32), rest.view(np.uint32))


def _level_exact(na, nk, ns, nc, eta):
    dt = np.sqrt(eta * (na * ns + nk * nk) / (nk * nc + ns * ns))
    return -(np.frexp(dt)[1] - 1)


def test_level_estimate_margin():
    # level_estimate of nb_device.cuh in numpy float32, with every operation's
    # result moved by up to two ulps (the device's approximate square roots and
    # division are that good): wherever it decides, it decides as the FP64
    # formulas do, also for norms placed so that dt_raw lies next to a power of two
    rng = np.random.RandomState(5)
    N = 400000

    def f32(x):
        y = np.asarray(x, dtype=np.float64).astype(np.float32)
        return (y * (1 + rng.randint(-2, 3, y.shape) * 2.0 ** -24)).astype(np.float32)

    na, nk, ns, nc = [10.0 ** rng.uniform(-6, 8, N) for _ in range(4)]
    eta = 0.01
    # the last half: scale the snap and crackle (dt ~ 1/scale) towards a binade edge
    dt = np.sqrt(eta * (na * ns + nk * nk) / (nk * nc + ns * ns))
    h = slice(N // 2, N)
    edge = 2.0 ** np.round(np.log2(dt[h])) * (1 + rng.choice([-1, 1], N // 2) * 10.0 ** rng.uniform(-9, -2, N // 2))
    lam = dt[h] / edge          # a, k, s, c scaled as 1, lam, lam^2, lam^3 divide dt by lam
    nk[h] *= lam
    ns[h] *= lam ** 2
    nc[h] *= lam ** 3
    n2 = [f32(f32(q) ** 2.0) for q in (na, nk, ns, nc)]
    n2 = [f32(q * (1 + rng.uniform(-3, 3, N) * 2.0 ** -24)) for q in n2]   # three-term sums
    root = [f32(np.sqrt(q.astype(np.float64))) for q in n2]
    num = f32(root[0].astype(np.float64) * root[2] + n2[1])
    den = f32(root[1].astype(np.float64) * root[3] + n2[2])
    with np.errstate(all="ignore"):
        R = f32(f32(eta * num.astype(np.float64)).astype(np.float64) / den)
        lo, hi = np.min(n2, axis=0), np.max(n2, axis=0)
        ok = (lo >= 2.0 ** -100) & (hi <= 2.0 ** 110) & (R >= 2.0 ** -72) & (R <= 2.0 ** 60)
    b = R.view(np.int32)
    e, m = (b >> 23) - 127, b & 0x7fffff
    ok &= np.where(e & 1, m < 0x800000 - 0x800, m >= 0x800)
    assert ok.mean() > 0.5 and not ok[h].all()
    assert np.array_equal(-(e >> 1)[ok], _level_exact(na, nk, ns, nc, eta)[ok])


def test_ticks_to_time_bits():
    # d 2^-40 built from the integer's bits
    rng = np.random.RandomState(6)
    d = np.concatenate([rng.randint(1, 1 << 53, 1000), 1 << np.arange(53), [(1 << 53) - 1, 3, 5]]).astype(np.int64)
    for q in d.tolist():
        sh = (64 - q.bit_length()) - 11
        bits = (q << sh) + ((1023 + 52 - 40 - 1 - sh) << 52)
        assert np.array([bits], dtype=np.uint64).view(np.float64)[0] == q * 2.0 ** -40


SRC_INT64 = r"""
#include <cstdio>
#include "nb_int64.cuh"
using namespace nbk::i64;
int main() {
    double a[6], c[6], m, e2, d[6], mr, mr3, b;
    for (;;) {
        for (int k = 0; k < 6; ++k) if (std::scanf("%lf %lf", a + k, c + k) != 2) return 0;
        if (std::scanf("%lf %lf", &m, &e2) != 2) return 0;
        Num D[6];
        bool ok = in_range(m) && eps2_in_range(e2);
        for (int k = 0; k < 6; ++k) {
            ok = ok && in_range(a[k]) && in_range(c[k]);
            D[k] = diff(to_fix(a[k]), to_fix(c[k]), d[k]);
        }
        pair_factors(D, D + 3, to_num(m), make_eps(e2), mr, mr3, b);
        for (int k = 0; k < 6; ++k) std::printf("%a ", d[k]);
        std::printf("%a %a %a %d\n", mr, mr3, b, ok ? 1 : 0);
    }
}
"""


def test_integer_pair_factors(tmp_path):
    # in units of 2^-53: a difference is rounded once (1, and 2^-8 for the cut);
    # r^2 loses at most 10 of 2^59 and so 1/r 0.08 more, its power 3 0.23, and the
    # products 3 of 2^60 each: 1.25, 1.5 and (of the sum of magnitudes) 1.5
    import os
    import shutil
    import subprocess
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src, exe = tmp_path / "i64.cpp", tmp_path / "i64"
    src.write_text(SRC_INT64)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + os.path.join(root, "paper_cs_0702135_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    rng = random.Random(3)
    rows = []
    for k in range(6000):
        wide = 99 if k % 3 == 0 else 6
        sx, sv = rng.uniform(-wide, wide), rng.uniform(-wide, wide)
        row = []
        for c in range(6):
            s = 2.0 ** min(99, max(-99, (sx if c < 3 else sv) + rng.uniform(-4, 4)))
            a, b = rng.uniform(-1, 1) * s, rng.uniform(-1, 1) * s
            b = rng.choice((b, b, 0.0, a, a * (1 + 2.0 ** -rng.randint(1, 52)), math.nextafter(a, 2 * a)))
            row += [a, b] if rng.random() < 0.5 else [b, a]
        if k % 50 == 0:
            row[6:] = [0.0] * 6
        if k % 60 == 0:
            row[:6] = [row[0]] * 6
        row += [rng.choice((0.0, 1.0, -1.0, 1.0)) * 2.0 ** rng.uniform(-99, 99),
                2.0 ** rng.uniform(-99, 99) if k % 2 else 2.0 ** rng.uniform(-20, -10)]
        rows.append(row)
    inp = "\n".join(" ".join(v.hex() for v in r) for r in rows)
    out = subprocess.run([str(exe)], input=inp, capture_output=True, text=True, check=True).stdout.splitlines()
    assert len(out) == len(rows)
    u, inside = F(1, 1 << 53), 0
    for row, line in zip(rows, out):
        got = [float.fromhex(t) for t in line.split()[:9]]
        if not int(line.split()[9]):
            continue   # too small a value: not taken by this arithmetic
        inside += 1
        d = [F(row[2 * c]) - F(row[2 * c + 1]) for c in range(6)]
        for c in range(6):
            assert abs(F(got[c]) - d[c]) <= abs(d[c]) * u * (1 + F(1, 256)), row
        r2 = sum(q * q for q in d[:3]) + F(row[13])
        num, den = r2.numerator << 600, r2.denominator << 600
        r = F(math.isqrt(num * den), den)
        m = F(row[12])
        assert abs(F(got[6]) - m / r) <= abs(m / r) * u * F(5, 4), row
        assert abs(F(got[7]) - m / r / r2) <= abs(m / r / r2) * u * F(3, 2), row
        dot = sum(d[c] * d[3 + c] for c in range(3))
        mag = sum(abs(d[c] * d[3 + c]) for c in range(3))
        assert abs(F(got[8]) + 3 * dot / r2) <= 3 * mag / r2 * u * F(3, 2), row
    assert inside > 5000

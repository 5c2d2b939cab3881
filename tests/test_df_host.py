"""Double-float arithmetic of the mixed refinement's residual products
(csrc/df.cuh), compiled for the host and checked against exact rational
arithmetic: the conversions from and to a double, and the paired sum,
difference, products and multiply-add within their derived error bounds, also
under cancellation.  These are the functions that the device passes run; only
the paired FP32 instructions below them are plain float operations here, each
rounded on its own on both sides."""
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0908_0863_gb300", "csrc")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
U2 = Fraction(2) ** -48        # square of a float's unit roundoff
SLACK = 1 + Fraction(2) ** -20   # third-order terms of the bounds


@pytest.fixture(scope="module")
def df_host(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs a host C++ compiler and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("df") / "df_host")
    subprocess.run([cxx, "-O2", "-std=c++17", "-w", "-ffp-contract=off", f"-I{CSRC}", f"-I{CUDA_INC}",
                    os.path.join(ROOT, "tests", "df_host.cpp"), "-o", exe], check=True)

    def run(op, rows):
        text = "".join(f"{op} {' '.join(float(v).hex() for v in row)}\n" for row in rows)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
        res = [[float.fromhex(w) for w in line.split()] for line in out if line]
        assert len(res) == len(rows)
        return res
    return run


def _pairs(x):
    """Doubles as rows (hi, lo) of the nearest float and the rounded remainder."""
    hi = x.astype(np.float32).astype(float)
    return np.stack([hi, (x - hi).astype(np.float32).astype(float)], axis=-1)


def _wide(rng, n):
    """Normalised pairs of random sign with magnitudes 2^-30..2^30."""
    return _pairs(rng.choice([-1.0, 1.0], n) * np.exp2(rng.uniform(-30, 30, n)))


def _near(rng, a):
    """Normalised pairs that nearly cancel a: minus a (1 + 2^-k u), k in 20..50,
    or the float of minus a's high part a few steps on, with a low part of up to
    half a last place (that of the low end exactly, at times)."""
    n = len(a)
    x = -(a[:, 0] + a[:, 1]) * (1.0 + np.exp2(-rng.integers(20, 51, n).astype(float)) * rng.uniform(-1, 1, n))
    b = _pairs(x)
    hi = (-a[:, 0]).astype(np.float32)
    for _ in range(3):
        step = rng.integers(-1, 2, n)
        hi = np.where(step < 0, np.nextafter(hi, np.float32(-np.inf)), np.where(step > 0, np.nextafter(hi, np.float32(np.inf)), hi))
    below = np.abs(hi.astype(float) - np.nextafter(hi, np.float32(0)).astype(float))   # last place towards zero
    part = rng.choice([-0.5, 0.5, 0.0, 1.0], n)
    lo = (np.where(part == 1.0, rng.uniform(-0.5, 0.5, n), part) * below).astype(np.float32).astype(float)
    steps = np.stack([hi.astype(float), lo], axis=-1)
    return np.where(rng.random(n)[:, None] < 0.5, b, steps)


def _edges(rng, n):
    """Pairs at both sides of a power of two, low parts up to half a last place."""
    hi = np.float32(2.0) ** rng.integers(-3, 4, n).astype(np.float32) * rng.choice([-1, 1], n).astype(np.float32)
    step = rng.integers(-1, 2, n)
    hi = np.where(step < 0, np.nextafter(hi, np.float32(0)), np.where(step > 0, np.nextafter(hi, np.float32(np.inf) * np.sign(hi)), hi))
    below = np.abs(hi.astype(float) - np.nextafter(hi, np.float32(0)).astype(float))
    lo = (rng.choice([-0.5, 0.5, 0.25, -0.25, 0.0], n) * below).astype(np.float32).astype(float)
    return np.stack([hi.astype(float), lo], axis=-1)


def _operands(kind, seed, n):
    rng = np.random.default_rng(seed)
    if kind == "wide":
        a, b, c = (np.concatenate([_wide(rng, n), _wide(rng, n)], axis=-1) for _ in range(3))
    elif kind == "edges":
        a, b, c = (np.concatenate([_edges(rng, n), _edges(rng, n)], axis=-1) for _ in range(3))
    else:
        a = np.concatenate([_wide(rng, n), _edges(rng, n)], axis=-1)
        b = np.concatenate([_near(rng, a[:, :2]), _near(rng, a[:, 2:])], axis=-1)
        c = np.concatenate([_near(rng, a[:, :2]), _near(rng, a[:, 2:])], axis=-1)
    return a, b, c


def _value(row, lane):
    return Fraction(float(row[2 * lane])) + Fraction(float(row[2 * lane + 1]))


def _normalised(row, lane):
    """hi is a float nearest hi + lo."""
    hi, lo = float(row[2 * lane]), Fraction(float(row[2 * lane + 1]))
    h = np.float32(hi)
    up, down = (Fraction(float(np.nextafter(h, np.float32(s)))) for s in (np.inf, -np.inf))
    return (Fraction(hi) - down) / 2 >= -lo and (up - Fraction(hi)) / 2 >= lo


KINDS = ["wide", "near", "edges"]


# ------------------------------------------------------------- conversions

def test_split_equals_the_conversion(df_host):
    rng = np.random.default_rng(1)
    exps = np.concatenate([rng.uniform(-30, 30, 300), rng.uniform(-74, -66, 300), rng.uniform(122, 127.9, 300),
                           rng.uniform(-160, -140, 100)])
    x = rng.choice([-1.0, 1.0], exps.size) * np.exp2(exps)
    b = x.view(np.uint64).copy()
    tie = rng.random(x.size) < 0.3            # low 29 bits exactly half a float's last place, and one either side
    b[tie] = (b[tie] & ~np.uint64(2**29 - 1)) + (2**28 + rng.integers(-1, 2, tie.sum())).astype(np.uint64)
    x = np.concatenate([b.view(np.float64), [0.0, -0.0, 1.0, 2.0 ** -70, 2.0 ** -71, 2.0 ** 126, -(2.0 ** 126),
                                             2.0 ** 127 * (1 - 2.0 ** -26), 5e-324]])
    for v, r in zip(x, df_host("split", x[:, None])):
        fast, conv = [Fraction(w) for w in r[:2]], [Fraction(w) for w in r[2:]]
        assert sum(fast) == sum(conv)
        half = (int(np.float64(v).view(np.uint64)) & (2**29 - 1)) == 2**28
        assert fast == conv or half
        if abs(v) >= 2.0 ** -100:
            assert abs(sum(fast) - Fraction(float(v))) <= U2 * abs(Fraction(float(v)))
            assert _normalised(r, 0)


def test_widen_is_exact(df_host):
    rng = np.random.default_rng(2)
    f = rng.integers(0, 2**32, 2000, dtype=np.uint64).astype(np.uint32).view(np.float32)
    f = f[np.isfinite(f)].astype(float)
    f = np.concatenate([f, [0.0, -0.0, 2.0 ** -126, 2.0 ** -149, -(2.0 ** -130), float(np.finfo(np.float32).max)]])
    for v, r in zip(f, df_host("widen", f[:, None])):
        assert r[0] == v and math.copysign(1.0, r[0]) == math.copysign(1.0, v)
    for v in (math.inf, -math.inf):
        assert df_host("widen", [[v]])[0][0] == v
    assert math.isnan(df_host("widen", [[math.nan]])[0][0])


# -------------------------------------------------------------- operations

@pytest.mark.parametrize("kind", KINDS)
def test_sum_and_difference(df_host, kind):
    # the low parts' sum rounds by at most u^2 (|a| + |b|), its sum with the
    # two-sum's error (each at most u (|a| + |b|)) by 2 u^2; the rest is exact
    a, b, _ = _operands(kind, 3, 1500)
    for op, sign in (("add", 1), ("sub", -1)):
        y = b if op == "add" else -b
        for x, z, r in zip(a, y, df_host(op, np.concatenate([a, y, y], axis=1))):
            for lane in (0, 1):
                p, q = _value(x, lane), _value(z, lane)
                assert abs(_value(r, lane) - (p + sign * q)) <= 3 * U2 * SLACK * (abs(p) + abs(q))
                assert _normalised(r, lane)


@pytest.mark.parametrize("kind", KINDS)
def test_products(df_host, kind):
    # ah bl and al bh are added to the exact error of ah bh with roundings of
    # 2 u^2 and 3 u^2, al bl (u^2) is dropped
    a, b, _ = _operands(kind, 4, 800)
    rows = np.concatenate([a, b, b], axis=1)
    for x, y, r, s in zip(a, b, df_host("mul2", rows), df_host("cscale", rows)):
        for lane in (0, 1):
            p, q, f = _value(x, lane), _value(y, lane), _value(y, 0)
            assert abs(_value(r, lane) - p * q) <= 6 * U2 * SLACK * abs(p * q)
            assert abs(_value(s, lane) - p * f) <= 6 * U2 * SLACK * abs(p * f)
            assert _normalised(r, lane) and _normalised(s, lane)


@pytest.mark.parametrize("kind", KINDS)
def test_complex_product_and_multiply_add(df_host, kind):
    # two products (6 u^2 each) and one or two sums (3 u^2 of their terms each)
    a, b, c = _operands(kind, 5, 800)
    rows = np.concatenate([a, b, c], axis=1)
    for x, y, z, r, s in zip(a, b, c, df_host("cmul", rows), df_host("cfma", rows)):
        xr, xi, yr, yi = _value(x, 0), _value(x, 1), _value(y, 0), _value(y, 1)
        for lane, (p, q) in enumerate(((xr * yr, -xi * yi), (xr * yi, xi * yr))):
            acc = _value(z, lane)
            assert abs(_value(r, lane) - (p + q)) <= 9 * U2 * SLACK * (abs(p) + abs(q))
            assert abs(_value(s, lane) - (acc + p + q)) <= 12 * U2 * SLACK * (abs(acc) + abs(p) + abs(q))
            assert _normalised(r, lane) and _normalised(s, lane)


def test_exact_cancellation_and_zero(df_host):
    one, tiny = _pairs(np.array([1.0 + 2.0 ** -30, -1.0])), _pairs(np.array([1.0 + 2.0 ** -40, -(1.0 + 2.0 ** -41)]))
    zero, three = [0.0, 0.0], [3.0, 0.0]
    r = df_host("add", [[*one[0], *tiny[0], *one[1], *tiny[1], *zero, *zero]])[0]
    # both operands carry their low parts: the differences are exact
    assert _value(r, 0) == Fraction(2) ** -30 and _value(r, 1) == Fraction(2) ** -41
    assert df_host("sub", [[*three, *zero, *three, *zero, *zero, *zero]])[0] == [0.0] * 4
    assert df_host("mul2", [[*zero, *three, *three, *zero, *zero, *zero]])[0] == [0.0] * 4
    assert df_host("cmul", [[*zero, *zero, *three, *three, *zero, *zero]])[0] == [0.0] * 4

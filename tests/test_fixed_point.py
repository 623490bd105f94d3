"""The integer-pipe arithmetic of mag_fx.cuh (host build of the same functions)
against integers and 60-digit decimals: squared distances exactly, distances
within 2^-60, exponentials within 0.55 units in the last place, over the limb
layouts and their edges; and the table against its generator."""
import ctypes
import os
import subprocess
import sys
from decimal import Decimal as D, getcontext

import numpy as np
import pytest

getcontext().prec = 60

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_23354_gb300", "csrc")

SHIM = r"""
#include "mag_fx.cuh"
using namespace mag;
static const fx_u64 T[FX_TABLE_SIZE] = {FX_TABLE_ENTRIES};
template <int LB> static void pairs(long n, int m, const long long* a, const long long* b, int e, double t, fx_u64* o) {
  const FxScale sc = fx_scale(t, e);
  for (long i = 0; i < n; ++i) {
    FxSquare q;
    FxSums s;
    fx_square_clear(q);
    fx_clear(s);
    for (int l = 0; l < m; ++l) {
      const long long x = a[i * m + l], y = b[i * m + l], mask = (1ll << LB) - 1;
      fx_accumulate(s, fx_coord{(int)(x & mask), (int)(x >> LB)}, fx_coord{(int)(y & mask), (int)(y >> LB)});
      if ((l + 1) % FX_SPILL == 0 || l + 1 == m) fx_add<LB>(q, s), fx_clear(s);
    }
    o[6 * i] = q.h, o[6 * i + 1] = q.l, o[6 * i + 2] = fx_close(q, m);
    if (fx_close(q, m)) continue;
    const FxRoot r = fx_root_start(q);
    const fx_u64 v = fx_root(r);
    o[6 * i + 3] = v, o[6 * i + 4] = (fx_u64)(long long)r.j;
    o[6 * i + 5] = fx_exp_neg(v, r.j - e + sc.kg, sc.g, T);
  }
}
extern "C" void fx_pairs(long n, int m, const long long* a, const long long* b, int e, double t, fx_u64* o) {
  fx_limb_of(m) == 31 ? pairs<31>(n, m, a, b, e, t, o) : pairs<30>(n, m, a, b, e, t, o);
}
extern "C" int fx_bits_of(int m) { return fx_coord_bits(m); }
extern "C" void fx_exps(long n, const fx_u64* d, const double* t, fx_u64* o, fx_u64* gs, int* kgs) {
  for (long i = 0; i < n; ++i) {
    fx_u64 g;
    int kg;
    fx_scale_t(t[i], &g, &kg);
    o[i] = fx_exp_neg_d(d[i], kg, g, T), gs[i] = g, kgs[i] = kg;
  }
}
extern "C" void fx_floats(long n, const double* d, double t, float* o) {
  fx_u64 g;
  int kg;
  fx_scale_t(t, &g, &kg);
  for (long i = 0; i < n; ++i) {
    union { double d; fx_u64 u; } x;
    x.d = d[i];
    int shift;
    const fx_u64 frac = (x.u & 0xfffffffffffffull) | 0x10000000000000ull;
    const fx_u64 z = fx_exp_fixed(frac << 10, (int)(x.u >> 52) - 1023 + kg, g, T, &shift);
    o[i] = fx_float_of(z, shift);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _ulps(bits, exact):
    """|value - exact| in units of the last place of the exact result."""
    got = D(float(np.uint64(bits).view(np.float64)))
    e = int(np.floor(float(exact.ln() / D(2).ln())))
    return abs(got - exact) / D(2) ** (e - 52)


@pytest.mark.parametrize("m", [1, 3, 4, 5, 16, 17, 33, 512])
@pytest.mark.parametrize("spread", [0, 12, 30])  # differences below 2^-spread of the range
def test_pairs(lib, m, spread):
    rng = np.random.default_rng(m * 100 + spread)
    bits, k, t = lib.fx_bits_of(m), 60, 1.7
    top = 2 ** bits - 1
    a = rng.integers(0, top, (k, m), dtype=np.int64)
    b = np.clip(a + rng.integers(-(2 ** (bits - spread)), 2 ** (bits - spread), (k, m)), 0, top)
    a[0], b[0] = 0, top  # the largest difference in every dimension
    e = bits - 3
    o = np.zeros((k, 6), np.uint64)
    lib.fx_pairs(ctypes.c_long(k), m, _ptr(a), _ptr(b), e, ctypes.c_double(t), _ptr(o))
    for i in range(k):
        q = sum((int(x) - int(y)) ** 2 for x, y in zip(a[i], b[i]))
        assert (int(o[i, 0]) << 64) | int(o[i, 1]) == q
        assert int(o[i, 2]) == ((q >> 64) < (m << 42))
        if o[i, 2]:
            continue
        d = D(q).sqrt() * D(2) ** -e
        s = D(int(o[i, 3])) * D(2) ** (-62 + int(o[i, 4].astype(np.int64)) - e)
        assert abs(s - d) <= d * D(2) ** -60
        z = (-D(t) * s).exp()  # of the distance as it was formed
        if z > D(2) ** -1000:
            assert _ulps(o[i, 5], z) <= D("0.55")


def test_exponential(lib):
    rng = np.random.default_rng(5)
    td = np.concatenate([rng.uniform(0, 64, 300), 10.0 ** rng.uniform(-18, 2.7, 300), np.arange(1, 64) * np.log(2) / 256])
    t = 10.0 ** rng.uniform(-3, 3, td.size)
    d = td / t
    o, g, kg = np.zeros(td.size, np.uint64), np.zeros(td.size, np.uint64), np.zeros(td.size, np.int32)
    lib.fx_exps(ctypes.c_long(td.size), _ptr(d), _ptr(t), _ptr(o), _ptr(g), _ptr(kg))
    for i in range(td.size):
        # t as it is taken: 256 t / ln 2 rounded to 64 bits
        ti = D(int(g[i])) * D(2) ** (int(kg[i]) - 63) * D(2).ln() / 256
        assert abs(ti - D(float(t[i]))) <= D(float(t[i])) * D(2) ** -64
        assert _ulps(o[i], (-ti * D(float(d[i]))).exp()) <= D("0.55")


# The FP32 entries of the batch's factor over every argument a pair can have: the
# pairs too close for the quantized coordinates come here whatever their t d.
# One rounding and the sticky bit's 2^-32; 0 (nothing else) from 2^-124 down.
def test_float_entries(lib):
    x = np.concatenate([np.linspace(1e-12, 90.0, 4001), 10.0 ** np.linspace(1.9, 12.0, 4001), [86.0, 88.7, 89.0, 1e6]])
    for t in (0.7, 1e5):
        d, o = np.ascontiguousarray(x / t), np.zeros(x.size, np.float32)
        lib.fx_floats(ctypes.c_long(d.size), _ptr(d), ctypes.c_double(t), _ptr(o))
        ref = np.exp(-(t * d).astype(np.longdouble))
        small = ref < 2.0 ** -123
        assert np.all(np.abs(o[~small] - ref[~small]) <= (2.0 ** -24 + 2.0 ** -30) * ref[~small])
        assert np.all((o[small] == 0.0) | (np.abs(o[small] - ref[small]) <= 2.0 ** -24 * ref[small] + 2.0 ** -148))


def test_table_is_generated():
    out = subprocess.run([sys.executable, os.path.join(CSRC, "gen_fx_table.py")], check=True, capture_output=True, text=True)
    with open(os.path.join(CSRC, "fx_table.inc")) as f:
        assert out.stdout == f.read()

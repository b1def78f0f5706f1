"""The fixed-point base-2 exponential and logarithm of the tile kernel
(csrc/pyro_fixed_math.cuh), compiled as host C++, against long double arithmetic.

Bounds from the formats: the exponential is rounded once to 53 bits (2^-53 relative)
after a series and three truncated products of 2^-64, each scaled by at most 2^-10:
3 2^-53; the logarithm is rounded to an even multiple of 2^-50 (error 2^-50) after a
series good to 2^-53: 1.2 2^-50; products of a coefficient and a factor drop the product
of the low halves (2^-2 units) and round: 1 unit of 2^-50 (a Horner step doubles it).
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_24286_gb300", "csrc")

PROGRAM = r"""
#include "pyro_fixed_math.cuh"
#include <cmath>
#include <cstdio>
#include <random>
using namespace pfx;
int main() {
  static u64 et[1024];
  static Log2Entry lt[256];
  for (int j = 0; j < 1024; ++j) et[j] = (u64)roundl(exp2l(j / 1024.0L) * 9223372036854775808.0L);
  for (int j = 0; j < 256; ++j) {
    lt[j].rc = (unsigned)roundl(2048.0L / (1.0L + (j + 0.5L) / 256));
    lt[j].L = (i64)llroundl(-log2l(lt[j].rc / 2048.0L) * 4611686018427387904.0L);
  }
  std::mt19937_64 g(7);
  const long double one = exp2l(50);
  double e = 0, l = 0, m = 0, h = 0, d = 0, edge = 0;
  for (int i = 0; i < 1000000; ++i) {
    i64 x = ((i64)(g() % (2000ull << 50)) - (1000ll << 50)) & ~1ll;
    if (i < 4096) x = ((i64)(i - 2048) << 40) + (i % 3 - 1) * 2;        // the ends of table cells
    const long double t = exp2l(x / one);
    e = fmax(e, (double)fabsl(exp2_lg(x, et) / t - 1));
    if (!(fabs(exp2_lg(x | 1, et) / -exp2_lg(x, et) - 1) <= 2.0 / one)) edge = 1;
    double v = bitsd((g() >> 12) | 0x3ff0000000000000ull);
    if (i < 512) v = 1.0 + (i / 2) / 256.0 - (i % 2 ? exp2(-52) : 0.0);
    if (v < 1.0) v = 1.0;
    v = ldexp(v, (int)(g() % 2000) - 1000);
    l = fmax(l, (double)fabsl(log2_of(v, lt) / one - log2l((long double)v)));
    const i64 c = (i64)g() / 2, f = (i64)((double)(g() >> 1) * 0.9999), q = (i64)g() / 4;
    m = fmax(m, (double)fabsl(mul_add(split(c), split(f), 0) - c / exp2l(51) * (f / exp2l(63)) * one));
    h = fmax(h, (double)fabsl(horner(q, split(f), 5) - 5 - q * (f / exp2l(63))));
    d = fmax(d, (double)fabsl(to_double(q) / (q / one) - 1));
    const double y = ldexp(1.0 + (g() >> 12) * exp2(-52), -1 - (int)(g() % 40)) * 0.9999;
    d = fmax(d, (double)(fabsl(frac_of(y) / exp2l(63) - y) / y - exp2l(-63) / y));
  }
  if (exp2_lg(LG_ZERO + (1190ll << 50), et) != 0.0 || !std::isinf(exp2_lg(1024ll << 50, et)) ||
      exp2_lg(-(1023ll << 50), et) != 0.0 || 3 * (LG_ZERO / 1024) < -(8192ll << 40)) edge = 1;
  printf("%.6g %.6g %.6g %.6g %.6g %g\n", e, l, m, h, d, edge);
}
"""


def test_exp2_log2_and_products(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "fixed.cpp"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(tmp_path / "fixed")], check=True)
    out = subprocess.run([str(tmp_path / "fixed")], capture_output=True, text=True, check=True).stdout.split()
    e, l, m, h, d, edge = map(float, out)
    assert e <= 3 * 2.0 ** -53
    assert l <= 1.2 * 2.0 ** -50
    assert m <= 1.0 and h <= 2.0
    assert d <= 2.0 ** -52
    assert edge == 0


def test_mechanisms_that_do_not_fit_the_tables_keep_the_fp64_kernel(mech_files, tmp_path):
    """The workload mechanisms use the tile kernel from 300 K or below; a fourth-order reaction or
    coefficients beyond the fixed-point range leave the handle on the FP64 kernel alone."""
    from paper_2503_24286_gb300 import binding as B
    from tests import handmech
    for i in (0, 1, 7):
        m = B.Mechanism(mech_files[0][i], "device=0")
        assert m.stat("tile") == 1 and m.stat("tile_t_lo") <= 300.0 and m.stat("tile_cubin_bytes") > 1000
    mech = handmech.abcd_mechanism()
    mech.reactions[0].reactants = [(0, 2), (1, 2)]
    mech.reactions[0].products = [(2, 2), (3, 2)]
    assert B.Mechanism(handmech.write(mech, str(tmp_path), "order4.txt"), "device=0").stat("tile") == 0
    mech = handmech.abcd_mechanism(theta=3.0e6)
    assert B.Mechanism(handmech.write(mech, str(tmp_path), "theta.txt"), "device=0").stat("tile") == 0


def test_the_tile_option(mech_files):
    """tile=0 leaves a handle on the FP64 kernels alone; other values are refused."""
    from paper_2503_24286_gb300 import binding as B
    m = B.Mechanism(mech_files[0][0], "device=0;tile=0")
    for key in ("tile", "jvp_tile", "vjp_tile", "jacobian_tile", "transport_tile"):
        assert m.stat(key) == 0
    assert B.Mechanism(mech_files[0][0], "device=0;tile=auto").stat("tile") == 1
    with pytest.raises(B.PyroError):
        B.Mechanism(mech_files[0][0], "device=0;tile=2")

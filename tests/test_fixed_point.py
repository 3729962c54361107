"""csrc/fx.cuh (the ALC screen's 64-bit fixed point) on the host against long double: the
header is plain integer code, compiled here with g++.  Bounds, in units of 2^-60 unless said
otherwise: 2^-y: 2 units in E, twice 2 in T E and 1 of T's truncation, 8 with the coefficients';
a correlation: those, y's truncations (40), and of the coordinates' own rounding by 2^-(59-b)
each, sum 2 |d_k| 2^-(58-b) ln 2 2^-y <= 5 2^b units in three dimensions; 1 / sqrt: 2^-57
relative; a factor entry (units of 2^-58): three truncations and 2 of 1 / sqrt; a product: one
truncation and the left-out low product, 2; a float: 2 ulp and the low word's rounding, 2^7."""
from __future__ import annotations

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "fx.cuh"
#include <cstdio>
#include <cstdlib>
#include <algorithm>
using namespace lagp;
typedef long double LD;
static uint64_t st = 88172645463325252ull;
static uint64_t rnd() { st ^= st << 13; st ^= st >> 7; st ^= st << 17; return st; }
int main() {
  const LD a = logl(2.0L) / 256;
  static uint64_t tab[256];
  for (int i = 0; i < 256; i++) tab[i] = (uint64_t)roundl(ldexpl(exp2l(-(LD)i / 256), 63));
  const uint64_t c1 = roundl(ldexpl(a, 60)), c2 = roundl(ldexpl(a * a / 2, 60));
  const uint32_t c3 = roundl(ldexpl(a * a * a / 6, 60)), c4 = roundl(ldexpl(a * a * a * a / 24, 60)),
                 c5 = roundl(ldexpl(a * a * a * a * a / 120, 60));
  LD ee = 0, er = 0, em = 0, ef = 0, ep = 0;
  for (int k = 0; k < 400000; k++) {
    // 2^-y over all magnitudes of y below 64, and its exact ends
    uint64_t Y = (rnd() >> 2) >> (rnd() % 62);
    if (k < 512) Y = (uint64_t)k << 48;
    else if (k < 1024) Y = ((uint64_t)(k - 511) << 48) - 1;
    const LD y = ldexpl((LD)Y, -56);
    ee = std::max(ee, fabsl((LD)fx_exp2(Y, tab, c1, c2, c3, c4, c5, 0) - ldexpl(exp2l(-y), 60)));
    // 1 / sqrt over every variance that the screen takes, 2^-30 .. 2
    const int64_t V = (int64_t)((rnd() | (1ull << 63)) >> (2 + rnd() % 31));
    const FxRsqrt r = fx_rsqrt(V);
    const LD nu = ldexpl((LD)V, -60);
    const LD R = ldexpl((LD)r.Rh * 4294967296.0L + r.Rl, -62 + r.q);
    er = std::max(er, fabsl(R * sqrtl(nu) - 1));
    // t / sqrt(nu), |t| <= sqrt(nu): factor entries, value 2^58
    const int64_t t = (int64_t)ldexpl(sqrtl(nu) * ((LD)(int64_t)rnd() / 9223372036854775808.0L), 60);
    const int64_t u = fx_mul_rsqrt(t, r);
    em = std::max(em, fabsl((LD)u - ldexpl(ldexpl((LD)t, -60) / sqrtl(nu), 58)));
    const FxU s = fx_split(u), w = fx_split((int64_t)rnd() >> 5);
    if ((int64_t)s.h * (1 << 28) + s.l != u) return 2;
    const LD p = ldexpl((LD)u * ((LD)w.h * 268435456.0L + w.l), -56);
    ep = std::max(ep, fabsl((LD)fx_mul_uu(s, w) - p));
    const int64_t x = (int64_t)rnd() >> (rnd() % 63);
    if (x) ef = std::max(ef, fabsl((LD)fx_to_float(x) - x) - 128 - 2 * ldexpl(fabsl((LD)x), -23));
  }
  // distances, from coordinates of every spread (b = 0 .. 8): relative to 1
  LD ed = 0;
  for (int k = 0; k < 200000; k++) {
    const int b = k % 9, e = 0;
    int64_t hh = 0, hl = 0, ll = 0;
    LD y = 0;
    const LD span = ldexpl(1.0L, (int)(rnd() % 12) - 12 + std::min(b, 3));
    for (int q = 0; q < 3; q++) {
      LD c[2];
      int32_t h[2], l[2];
      for (int i = 0; i < 2; i++) {
        c[i] = span * ((LD)(int64_t)rnd() / 9223372036854775808.0L) * (b ? 1.0L : 0.9L);
        const LD s = ldexpl(c[i], 28 - b);
        h[i] = (int32_t)rintl(s);
        l[i] = (int32_t)rintl(ldexpl(s - h[i], 30));
      }
      const int64_t dh = h[0] - h[1], dl = l[0] - l[1];
      hh += dh * dh; hl += dh * dl; ll += dl * dl;
      y += (c[0] - c[1]) * (c[0] - c[1]);
    }
    const LD bound = 8 + 40 + 5 * ldexpl(1.0L, b);
    ed = std::max(ed, fabsl((LD)fx_corr(hh, hl, ll, 2 * b, tab, c1, c2, c3, c4, c5, e) -
                            ldexpl(y < 64 ? exp2l(-y) : 0.0L, 60)) / bound);
  }
  printf("exp %Lg units, rsqrt %Lg, entry %Lg units, product %Lg units, float %Lg past its bound, corr %Lg of its bound\n",
         ee, er * ldexpl(1, 57), em, ep, ef, ed);
  return ee <= 8 && er * ldexpl(1, 57) <= 1 && em <= 5 && ep <= 2 && ef <= 0 && ed <= 1 ? 0 : 1;
}
"""


def test_fixed_point_against_long_double(tmp_path):
    src = tmp_path / "fx.cpp"
    src.write_text(SRC)
    exe = tmp_path / "fx"
    subprocess.run(["g++", "-O1", "-x", "c++", "-I", os.path.join(ROOT, "paper_1303_0383_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    print(r.stdout)
    assert r.returncode == 0, r.stdout

"""The float-pair arithmetic of the double-precision near field (csrc/ff64.cuh),
compiled for the host and compared with 40-digit values: the pair terms
q ln r^2 and q (dx, dy) / r^2 formed from fixed-point coordinates, at the edges
of the coordinate, exponent and charge ranges, and the three-float sum.

Tolerances from the arithmetic: a pair (h, l) holds 2^-49 relative; dx adds
one such rounding, r^2 doubles it and adds three, ln r^2 adds four of at most
2^-50 absolute to r^2's relative error, the reciprocal two and the products
three more: 2^-45 bounds each with a factor of two to spare."""
import os
import subprocess

import numpy as np
import pytest

mpmath = pytest.importorskip("mpmath")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_21913_gb300", "csrc")
TOL = 2.0 ** -45

HARNESS = r"""
#include <stdio.h>
#include "ff64.cuh"
int main() {
  static ff tab[kFfLogN];
  ff_log_table(tab);
  double x, y, x2, y2, q;
  int kd, down, nudge;
  while (scanf("%la %la %la %la %la %d %d %d", &x, &y, &x2, &y2, &q, &kd, &down, &nudge) == 8) {
    const int s = 60 - kd;
    const ff dx = ff_from_fixed(ff_fixed(x, s) - ff_fixed(x2, s));
    const ff dy = ff_from_fixed(ff_fixed(y, s) - ff_fixed(y2, s));
    const ff w = ff_split_scaled(q, down), r2 = ff_norm2(dx, dy);
    const float c = ff_from(ff_bits(1.0f / r2.h) + nudge);
    float k;
    const ff m = ff_log(r2, c, tab, 46 - 2 * kd, k);
    const ff qw = ff_prod(ff_recip(r2, c), w), gx = ff_prod(qw, dx), gy = ff_prod(qw, dy);
    printf("%a %a %a %a %a %a %a %a\n", (double)k, (double)m.h + m.l, (double)gx.h, (double)gx.l,
           (double)gy.h, (double)gy.l, (double)w.h, (double)w.l);
  }
  // sums of a long alternating series: the last line
  ff_sum3 t{0, 0, 0};
  for (int i = 0; i < 20000; ++i) {
    const float v = ldexpf((float)((i * 7919) % 1000 - 499.5f), i % 40 - 20);
    t.add(ff{v, v * 1e-8f});
    t.add(ff{-v, v * 1e-9f});
  }
  printf("%a\n", t.value());
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("ff64")
    (d / "h.cpp").write_text(HARNESS)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC,
                        str(d / "h.cpp"), "-o", str(d / "h")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "h")


def _samples(rng, kind):
    for i in range(400):
        kd = int(rng.integers(-12, 4)) if kind != "far side" else int(rng.choice([-300, 200]))
        d = 2.0 ** kd * rng.uniform(0.51, 1.0)
        # a coordinate of the grid's magnitude (its double has few spare bits)
        x, y = (rng.random(2) if kind != "far side" else rng.random(2) * d * 4)
        sep = 2 * d * 2.0 ** -rng.uniform(0, 26 if kind == "close" else 3)
        th = rng.uniform(0, 2 * np.pi) if i % 5 else (i % 4) * np.pi / 2
        if kind == "axis":  # one difference zero (never both: the kernel takes those apart)
            th = (1 if i % 2 else -1) * np.pi / 2
        x2, y2 = x + sep * np.cos(th), y + sep * np.sin(th)
        q = rng.uniform(-1, 1) * 2.0 ** (0 if i % 7 else -40)
        if kind == "axis":
            x2 = x
        yield x, y, x2, y2, q, kd, 0, i % 3 - 1


@pytest.mark.parametrize("kind", ["ordinary", "close", "axis", "far side"])
def test_pair_terms(harness, kind):
    rng = np.random.default_rng(3)
    rows = list(_samples(rng, kind))
    inp = "\n".join(" ".join([float(v).hex() for v in r[:5]] + [str(v) for v in r[5:]])
                    for r in rows) + "\nend\n"
    out = subprocess.run([harness], input=inp, capture_output=True, text=True, check=True).stdout
    lines = out.strip().split("\n")
    assert len(lines) == len(rows) + 1
    mp = mpmath.mp
    mp.dps = 40
    for r, line in zip(rows, lines):
        x, y, x2, y2, q, kd, _, _ = r
        k, m, gxh, gxl, gyh, gyl, wh, wl = (float.fromhex(t) for t in line.split())
        unit = mp.mpf(2) ** (kd - 60)
        # the coordinates as the kernel holds them: to the nearest unit
        dx = (mp.nint(mp.mpf(x) / unit) - mp.nint(mp.mpf(x2) / unit)) * unit
        dy = (mp.nint(mp.mpf(y) / unit) - mp.nint(mp.mpf(y2) / unit)) * unit
        r2 = dx * dx + dy * dy
        w = mp.mpf(wh) + wl
        assert abs(w - q) <= 2.0 ** -48 * abs(q)
        assert abs(m) < 0.4 and k == int(k)
        assert abs(k * mp.log(2) + m - mp.log(r2)) < TOL
        scale = abs(w) / mp.sqrt(r2)
        g = mp.mpf(2) ** (23 - kd)  # the kernel's units
        assert abs(g * (mp.mpf(gxh) + gxl) - w * dx / r2) < TOL * scale
        assert abs(g * (mp.mpf(gyh) + gyl) - w * dy / r2) < TOL * scale


def test_three_float_sum(harness):
    out = subprocess.run([harness], input="end\n", capture_output=True, text=True,
                         check=True).stdout
    got = float.fromhex(out.strip())
    f = np.float32
    ref, big = mpmath.mpf(0), 0.0
    for i in range(20000):
        v = f(np.ldexp(f((i * 7919) % 1000 - 499.5), i % 40 - 20))
        big = max(big, abs(float(v)))
        ref += mpmath.mpf(float(f(v * f(1e-8)))) + mpmath.mpf(float(f(v * f(1e-9))))
    # each term adds at most its own 2^-48; the running sum adds 2^-70 of itself
    assert abs(got - ref) < 40000 * 2.0 ** -49 * 1e-7 * big + 2.0 ** -46 * abs(ref)

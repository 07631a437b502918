"""The integer arithmetic of the double-precision near field (csrc/fix64.cuh),
compiled for the host and compared with 40-digit values of the pair terms
q ln r^2 and q (dx, dy) / r^2 of the coordinates' and charges' true doubles.

Bounds.  The integers of a gradient term (R, 1 / R, q / R, q x / R) are off by at
most 5, 3, 4 and 4 units of at least 2^60, 2^59, 2^57 and 2^56.5, together below
2^-53.5 of |q| / r; a coordinate's unit, 2^-92, adds 2^-80 at the least distance.
ln r^2 is off by 2^-57 for R, 2^-55 for the series, by two units of the scale that
holds the largest logarithm (2^-57 of it) and by the product's four: below 2^-53 of
max(1, |ln r^2|) where the scale is within 8 of it.  The value read out is rounded
to 53 bits once more."""
import os
import subprocess

import numpy as np
import pytest

mpmath = pytest.importorskip("mpmath")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_21913_gb300", "csrc")

HARNESS = r"""
#include <stdio.h>
#include "fix64.cuh"
int main(int argc, char **argv) {
  static int64_t plain[kFfLogN], tab[kFfLogN];
  fx_log_table(plain);
  double x, y, x2, y2, q;
  int kd, emax, nudge;
  FxSums all;
  all.clear();
  while (scanf("%la %la %la %la %la %d %d %d", &x, &y, &x2, &y2, &q, &kd, &emax, &nudge) == 8) {
    const int s = 60 - kd;
    const fx96 dx = fx_sub(fx_fixed(x, s), fx_fixed(x2, s));
    const fx96 dy = fx_sub(fx_fixed(y, s), fx_fixed(y2, s));
    const uint32_t reach = fx_reach(dx, dy);
    const FxCharge w = fx_charge(q, emax);
    const FxScale c = fx_scale(kd);
    for (int i = 0; i < kFfLogN; ++i) tab[i] = c.tab(plain[i]);
    FxSums a;
    a.clear();
    if (reach >= fx_cut(w.drop)) {
      fx_pair(a, dx, dy, reach, w.bits, w.drop, c, tab, nudge);
      fx_pair(all, dx, dy, reach, w.bits, w.drop, c, tab, nudge);
    }
    printf("%d %a %a %a\n", reach >= fx_cut(w.drop), a.log_sum(emax, c), a.gx(emax, kd), a.gy(emax, kd));
  }
  printf("%a %a %a\n", all.x.value(0), all.y.value(0), all.l.value(0));
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("fix64")
    (d / "h.cpp").write_text(HARNESS)
    # undefined behaviour (a shift or a signed sum out of range) ends the run
    r = subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=undefined",
                        "-fno-sanitize-recover=undefined", "-I", CSRC, str(d / "h.cpp"), "-o",
                        str(d / "h")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "h")


def run(harness, rows):
    inp = "\n".join(" ".join([float(v).hex() for v in r[:5]] + [str(v) for v in r[5:]])
                    for r in rows) + "\nend\n"
    out = subprocess.run([harness], input=inp, capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    return [line.split() for line in out.stdout.strip().split("\n")]


def samples(rng, kind, count=600):
    for i in range(count):
        kd = int(rng.integers(-14, 3))
        if kind == "far scale":
            kd = int(rng.choice([-900, -300, 200, 900]))
        d = 2.0 ** kd * rng.uniform(0.51, 1.0)  # the leaf side
        sep = 2 * d * 2.0 ** -rng.uniform(0, 2 if kind == "wide" else 12.9)
        th = rng.uniform(0, 2 * np.pi) if i % 5 else (i % 4) * np.pi / 2
        x, y = rng.random(2) if kind != "far scale" else rng.random(2) * d * 4
        if kind == "shifted":
            x += 700.0
        x2, y2 = x + sep * np.cos(th), y + sep * np.sin(th)
        if kind in ("axis", "corner"):
            # next to y = 0 (and x = 0): doubles finer than any fixed unit
            y, y2 = np.abs([rng.uniform(0, 1), rng.uniform(0, 1)]) * sep
            if i % 2:
                y *= 2.0 ** -rng.uniform(0, 60)
            if kind == "corner":
                x, x2 = np.array([rng.uniform(-1, 1), rng.uniform(-1, 1)]) * sep
                x *= 2.0 ** -rng.uniform(0, 60)
        if kind == "column":
            x2 = x
        q = rng.uniform(-1, 1) * 2.0 ** -rng.choice([0, 0, 5, 16, 17, 18, 26])
        yield x, y, x2, y2, q, kd, 1022, i % 3 - 1


@pytest.mark.parametrize("kind", ["wide", "ordinary", "shifted", "axis", "corner", "column",
                                  "far scale"])
def test_pair_terms(harness, kind):
    rng = np.random.default_rng(11)
    rows = list(samples(rng, kind))
    lines = run(harness, rows)
    assert len(lines) == len(rows) + 1
    mp = mpmath.mp
    mp.dps = 60
    seen = 0
    for r, line in zip(rows, lines):
        x, y, x2, y2, q, kd = r[:6]
        if int(line[0]) == 0:
            continue
        seen += 1
        lv, gx, gy = (mp.mpf(float.fromhex(t)) for t in line[1:])
        dx, dy, w = mp.mpf(x) - mp.mpf(x2), mp.mpf(y) - mp.mpf(y2), mp.mpf(q)
        r2 = dx * dx + dy * dy
        ln = mp.log(r2)
        # the returned doubles are rounded once; weak charges count as 2^-17
        weak = max(abs(w), mp.mpf(2) ** (1022 - 1023 - 17))
        g = weak / mp.sqrt(r2)
        tol = mp.mpf(2) ** -53
        assert abs(gx - w * dx / r2) <= tol * (g + abs(gx))
        assert abs(gy - w * dy / r2) <= tol * (g + abs(gy))
        assert abs(lv - w * ln) <= tol * (weak * max(1, abs(ln)) + abs(lv))
    assert seen > len(rows) // 2


def test_charges(harness):
    """Weak charges down to zero, at every scale of the largest."""
    rng = np.random.default_rng(12)
    rows = []
    for drop in (0, 1, 16, 17, 18, 26, 27, 28, 60, 79, 100):
        for e in (1022, 140, 2000):
            m = 1.0 + rng.random()
            rows.append((0.3, 0.4, 0.35, 0.45, float(np.ldexp(m, e - 1023 - drop)), -3, e, 0))
    rows.append((0.3, 0.4, 0.35, 0.45, 0.0, -3, 1022, 0))
    lines = run(harness, rows)
    mp = mpmath.mp
    mp.dps = 60
    for r, line in zip(rows, lines):
        q, e = mp.mpf(r[4]), r[6]
        dx, dy = mp.mpf(r[0]) - mp.mpf(r[2]), mp.mpf(r[1]) - mp.mpf(r[3])
        r2 = dx * dx + dy * dy
        weak = max(abs(q), mp.mpf(2) ** (e - 1023 - 17))
        got = mp.mpf(float.fromhex(line[2]))
        assert abs(got - q * dx / r2) <= mp.mpf(2) ** -53 * (weak / mp.sqrt(r2) + abs(got))
    assert [float.fromhex(t) for t in lines[len(rows) - 1][1:]] == [0.0, 0.0, 0.0]


def test_sums_are_exact(harness):
    """Terms of both signs that cancel to nothing leave nothing, whatever lies
    between them, and a long sum equals the sum of its terms."""
    rng = np.random.default_rng(13)
    rows = list(samples(rng, "ordinary", 2000))
    rows = [r[:5] + (-3, 1022, 0) for r in rows]
    rows = [(r[0], r[1], r[0] + (r[2] - r[0]) % 0.1, r[1] + (r[3] - r[1]) % 0.1) + r[4:] for r in rows]
    back = [r[:4] + (-r[4],) + r[5:] for r in rows]
    rng.shuffle(back)
    lines = run(harness, rows + [tuple(b[:5]) + (int(b[5]), int(b[6]), int(b[7])) for b in back])
    total = [float.fromhex(t) for t in lines[-1]]
    # a product and its negative floor differently: one unit of 2^0 .. 2^31 a term
    assert all(abs(t) <= 4 * 4000 * 2.0 ** 31 for t in total)
    one = run(harness, rows)
    mp = mpmath.mp
    got = mp.mpf(float.fromhex(one[-1][0])) * mp.mpf(2) ** (1022 - 1023 + 3 - 77)
    ref = sum(mp.mpf(float.fromhex(line[2])) for line in one[:-1])
    big = sum(abs(float.fromhex(line[2])) for line in one[:-1])
    assert abs(got - ref) <= 2.0 ** -53 * big

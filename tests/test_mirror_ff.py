"""The float-pair form of the image and reaction pair (csrc/mirror_ff.cuh),
compiled for the host and compared with 40-digit values of Eqs. reactioncomp1,
reactioncomp2 over its range |P| <= 1/8: real and lossy kappa, pairs on the
axis, and down to 2^-14 of the range.

Each result is one rounding of a value good to 2^-36 of the potential's or the
gradient's magnitude, so it may be off by 2^-24 of itself and 2^-36 of that."""
import math
import os
import subprocess

import numpy as np
import pytest

mpmath = pytest.importorskip("mpmath")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_21913_gb300", "csrc")

HARNESS = r"""
#include <stdio.h>
#include "mirror_ff.cuh"
int main() {
  static ff lt[kFfLogN];
  static FfAngle at[kFfAng];
  ff_log_table(lt);
  ff_angle_table(at);
  double X, Y, kr, ki, lk, ak;
  while (scanf("%la %la %la %la %la %la", &X, &Y, &kr, &ki, &lk, &ak) == 6) {
    const KappaFF K{ff_of(kr), ff_of(ki), ff_of(lk), ff_of(ak), ki == 0};
    float v[6];
    ff_mirror((float)X, (float)Y, K, atan2f(fabsf((float)X), (float)Y), lt, at, v);
    for (int e = 0; e < 6; ++e) printf("%a ", (double)v[e]);
    printf("\n");
  }
  return 0;
}
"""


def reference(X, Y, kr, ki):
    mp = mpmath.mp
    mp.dps = 40
    X, Y, k = mp.mpf(X), mp.mpf(Y), mp.mpc(kr, ki)

    def J(P):
        Ei = mp.euler + mp.log(P) + sum(P ** n / (n * mp.factorial(n)) for n in range(1, 30))
        j = mp.e ** (-P) * (1j * mp.pi - Ei)
        return j, 1 + P * j
    sp, sm = mp.mpc(Y, -X), mp.mpc(Y, X)
    a, a1 = J(k * sp)
    b, b1 = J(k * sm)
    R2 = X * X + Y * Y
    u = (mp.log(R2) / 2 + a + b) / (2 * mp.pi)
    gx = (X / R2 + 1j * (a1 / sp - b1 / sm)) / (2 * mp.pi)
    gy = (Y / R2 - (a1 / sp + b1 / sm)) / (2 * mp.pi)
    g = mp.sqrt(abs(gx) ** 2 + abs(gy) ** 2)
    return [u.real, u.imag, gx.real, gx.imag, gy.real, gy.imag], [abs(u)] * 2 + [g] * 4


@pytest.mark.parametrize("loss", [0.0, 0.5])
def test_pair_values(tmp_path, loss):
    (tmp_path / "h.cpp").write_text(HARNESS)
    exe = str(tmp_path / "h")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC,
                        str(tmp_path / "h.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    rng = np.random.default_rng(1)
    rows = []
    for i in range(400):
        kr = float(rng.choice([1.0, 0.3, 5.0]))
        ki = loss * kr
        d = 0.1249 / abs(complex(kr, ki)) * 2.0 ** -rng.uniform(0, 14 if i % 3 else 0.01)
        th = rng.uniform(-1, 1) * np.pi / 2 * (1 - 1e-6) if i % 9 else 0.0
        rows.append((float(np.float32(d * np.sin(th))), float(np.float32(d * np.cos(th))), kr, ki,
                     0.5 * math.log(kr * kr + ki * ki), math.atan2(ki, kr)))
    inp = "\n".join(" ".join(float(v).hex() for v in row) for row in rows) + "\n"
    out = subprocess.run([exe], input=inp, capture_output=True, text=True, check=True).stdout
    lines = out.strip().split("\n")
    assert len(lines) == len(rows)
    for row, line in zip(rows, lines):
        ref, scale = reference(*row[:4])
        for v, e, s in zip((float.fromhex(w) for w in line.split()), ref, scale):
            assert abs(v - e) <= 2.0 ** -24 * abs(e) + 2.0 ** -36 * s

"""The fixed-point Hankel evaluator, compiled for the host, against mpmath over its
whole range: the device runs the same integer operations."""
import os
import subprocess

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2607_00790_gb300", "csrc")
MAIN = """
#include <cstdio>
#include "hankel_fixed.cuh"
int main() {
  static const HxNear near_ = {HX_NEAR_LO, HX_NEAR, HX_NEAR_SH};
  double z, u;
  while (scanf("%la %la", &z, &u) == 2) {
    HxUnit h;
    hankel_fixed(near_, z, u, h);
    printf("%a %a %a %a\\n", h.r0, h.i0, h.r1, h.i1);
  }
}
"""


def evaluate(z, u, tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", SRC, "-o", exe, str(tmp_path / "main.cpp")], check=True)
    out = subprocess.run([exe], input="\n".join(f"{float(a).hex()} {float(b).hex()}" for a, b in zip(z, u)), capture_output=True, text=True, check=True)
    v = np.array([[float.fromhex(t) for t in line.split()] for line in out.stdout.splitlines()])
    return v[:, 0] + 1j * v[:, 1], v[:, 2] + 1j * v[:, 3]


@pytest.mark.parametrize("ulps", [0, -4, 4])
def test_matches_mpmath(ulps, tmp_path):
    """Every component within its own rounding to double, 2^-58 (the fixed-point sums) and the
    change that the error of the 1/z given makes (|dP/du|, |dQ/du| <= 3/8)."""
    mp = pytest.importorskip("mpmath")
    rng = np.random.default_rng(0)
    bounds = np.array([1.5, 1.75, 2.0, 2.5, 3.25, 4.25, 5.75, 8.0, 12.0, 20.0])
    z = np.concatenate([
        np.exp(rng.uniform(np.log(1.5), np.log(2.0**20), 300)), rng.uniform(1.5, 20.0, 300),
        bounds, np.nextafter(bounds[1:], 0.0), np.nextafter(bounds, 99.0), [np.nextafter(2.0**20, 0.0)],
        2.0 ** np.arange(5, 20), np.nextafter(2.0 ** np.arange(5, 20), 0.0),
        20.0 + np.pi / 4 * np.arange(100),  # quadrant boundaries and zeros of a component
    ])
    u = 1.0 / z
    u = u + ulps * np.spacing(u)
    with mp.workdps(40):
        for nu, h in enumerate(evaluate(z, u, tmp_path)):
            for x, w, v in zip(z, u, h):
                x = mp.mpf(float(x))
                ref = mp.hankel1(nu, x) * mp.sqrt(mp.pi * x / 2)
                slack = mp.mpf(2) ** -58 + abs(mp.mpf(float(w)) - 1 / x) * 3 / 8
                for got, want in ((v.real, mp.re(ref)), (v.imag, mp.im(ref))):
                    assert abs(mp.mpf(float(got)) - want) <= abs(want) * mp.mpf(2) ** -53 + slack, (nu, x)

"""The 1D integrator's fixed-point arithmetic on the host (the functions that
the kernel compiles, no GPU): the guard of its range, and its rounding."""
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1105_4840_gb300 import build, pmf


@pytest.mark.parametrize("X,outside", [(0, False), (2**62 - 1, False), (-2**62, False), (2**62, True), (-2**62 - 1, True),
                                       (2**62 + 2**32, True), (2**63 - 1, True), (-2**63, True)])
def test_guard_sees_every_position_outside(X, outside):
    """Without a force, from 0, the position is q."""
    pos, out = pmf.pmf_od1d_fixed_map(0.0, 0.0, 0, 0, [X])
    assert pos[0] == X and out is outside


@pytest.mark.parametrize("sign", [1, -1])
def test_guard_keeps_what_it_saw(sign):
    """Out of the range for one step only, and back."""
    q = np.array([sign * 2**61, sign * 2**61 + sign, -sign * 2**62, 5])
    pos, out = pmf.pmf_od1d_fixed_map(0.0, 0.0, 0, 0, q)
    assert list(pos) == list(np.cumsum(q)) and out


PROGRAM = r"""
#include "fixed62.h"
int main()
{
    const long long top = 0x7fffffffffffffffLL, q[] = {0, 1LL << 62, -(1LL << 62) - 1, top, -top - 1, (1LL << 62) - 1};
    unsigned bits = 0;
    for (int i = 0; i < 6; ++i) bits |= (pmf::range_guard(q[i]) >> 31) << i;
    // positions inside the range, each factor of a step near its limit
    const pmf::FixedStep f{pmf::limbs(-((1LL << 62) - 1)), (1LL << 62) - 1};
    long long x = -(1LL << 61);
    for (int i = 0; i < 4; ++i) x = pmf::fixed_step(f, x, 12345) / 4;
    return bits == 0x1e && (pmf::range_guard(x) >> 31) == 0 ? 0 : 1;
}
"""


def test_no_undefined_overflow(tmp_path):
    """The guard and a step under the host compiler's overflow checks: a
    position above the range must not be found by an overflow that the compiler may assume
    away."""
    src, exe = tmp_path / "guard.cpp", tmp_path / "guard"
    src.write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which(build._nvcc()) or "/usr/local/cuda/bin/nvcc")), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-D__forceinline__=inline", "-I", build.CSRC, "-I", cuda, "-fsanitize=undefined",
                    "-fno-sanitize-recover=all", str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


# double well, weak well, trap alone (small, large and dyadic coefficients), inverted well
@pytest.mark.parametrize("a,k,dt,b", [(2.0, 20.0, 1e-3, 2), (2.0, 0.1, 1e-3, 3), (0.01, 1.0, 1e-3, 4), (0.0, 1.0, 1e-3, 4),
                                      (0.0, 20.0, 1e-5, 0), (0.0, 1e8, 1e-9, -8), (0.0, 1.0, 2.0**-10, 4), (0.0, 2.0, 0.05, 3),
                                      (-0.1, 1.0, 5e-3, 2)])
def test_steps_round_to_either_side(a, k, dt, b):
    """Every step against its exact image of the position before it.  A step's
    error has a variance below 1.4 units^2 (two cross products of 1/3 each, the
    low limbs 0.05, the split of the offset 0.25, w's own 1.1 at |x| <= 0.6 of the range), so the
    mean over N steps stays within 5 sqrt(1.4 / N); beside that the offset of w is a whole
    number, at most 1/2 off, which x < 2^62 multiplies, and q's has 1/256 units
    (the dyadic coefficient's cross products miss another 2^-11 each)."""
    cA, cB1, N = -4.0 * a * dt, (4.0 * a - k) * dt, 20000
    g = np.random.default_rng(4)
    amp = 0.07 * math.sqrt(2 * dt * k) * 2.0**62  # stationary width 0.07 of the range without wells
    q = np.array([int(v) for v in np.clip(g.normal(0.0, amp, N), -2.0**60, 2.0**60)], dtype=np.int64)
    q += g.integers(-512, 512, N)
    X, out = pmf.pmf_od1d_fixed_map(cA, cB1, b, 2**59, q)
    assert not out and np.abs(X).max() < 0.6 * 2.0**62
    fA, fB = Fraction(cA) * Fraction(4) ** b, Fraction(cB1)
    err, x0 = 0.0, 2**59
    for x1, qn in zip(X.tolist(), q.tolist()):
        x = Fraction(x0, 2**62)
        e = x1 - (x0 + qn + x0 * (fB + fA * x * x))
        assert abs(e) < 8
        err += float(e)
        x0 = x1
    assert abs(err / N) <= 5 * math.sqrt(1.4 / N) + 0.5 * abs(X.astype(float).mean()) / 2.0**62 + 2 / 256

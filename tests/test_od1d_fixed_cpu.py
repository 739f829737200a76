"""The 1D integrator's fixed-point arithmetic on the host (the functions that
the kernel compiles, no GPU): the guard of its range, its rounding, and the
choice of the range."""
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


def test_range_holds_the_motion_and_keeps_fp64s_precision():
    """Over many models and traps: the range holds what it must, no step from
    inside can wrap, and its unit stays below FP64's rounding of |x|, 2^b <= 128 |x| (the
    error of a step is 1.2 units of 2^(b-62), FP64's |x| 2^-53.7)."""
    g = np.random.default_rng(12)
    taken = 0
    for _ in range(20000):
        a = float(g.choice([0.0, 2.0, 10 ** g.uniform(-6, 2), -(10 ** g.uniform(-3, 0))]))
        x0, k, kT = float(g.normal(0, 1)), 10 ** g.uniform(-3, 8), 10 ** g.uniform(-4, 2)
        dt = float(10 ** g.uniform(-6, 0) / (k + 8 * abs(a)))
        far = float(abs(g.normal()) * 10 ** g.uniform(-2, 9))
        near = float(far * g.choice([0.0, 1.0, g.random()]))
        b = pmf.pmf_od1d_range(a, x0, k, kT, dt, 1.0, far, near)
        if b is None:
            continue
        taken += 1
        s, amp = math.sqrt(kT / k), math.sqrt(2 * kT * dt)
        assert 2.0**b >= max(far, abs(x0), a != 0) + 6 * s
        size = max(math.sqrt(kT / (k + 4 * abs(a))), near if a == 0 else min(near, 1.0) if a > 0 else 0.0)
        assert 2.0**b <= 128 * size
        assert abs(4 * a - k) * dt + abs(4 * a * dt) * 4.0**b + (6.8 * amp + k * dt * far) / 2.0**b < 1.0
    assert taken > 2000


@pytest.mark.parametrize("far,b", [(1.5, 2), (0.0, 2), (2.6, 2), (2.8, 3), (100.0, None)])
def test_range_of_the_double_well(far, b):
    assert pmf.pmf_od1d_range(2.0, -1.0, 20.0, 1.0, 1e-3, 1.0, far, far) == b

"""The 1D integrator's fixed-point arithmetic on the host (the functions that
the kernel compiles, no GPU): the guard of its range."""
import os
import shutil
import subprocess

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

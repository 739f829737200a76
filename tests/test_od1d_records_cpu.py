"""Which records the 1D integrator's helper warps take, and when (host side of
the kernel's own walk, no GPU): every record number once, by helper number
mod 3, at the end of step n_equil + (at + 1) stride - 1, up to the largest
stride and step count the API takes."""
import numpy as np
import pytest

from paper_1105_4840_gb300 import pmf


@pytest.mark.parametrize("stride", [1, 2, 7, 40, 1000, 715_827_882, 715_827_883, 2**30, 2**31 - 1])
@pytest.mark.parametrize("n_equil,start", [(0, 0), (5, 0), (5, 6), (123, 8160), (2**31, 2**32 - 41)])
def test_records_of_the_helpers(stride, n_equil, start):
    n = 5
    first = max(start - n_equil, 0) // stride  # records before step `start`
    got = sorted(zip(*map(np.ndarray.tolist, map(np.concatenate, zip(
        *(pmf.pmf_od1d_records(h, n_equil, stride, start, n) for h in range(3)))))))
    assert got == [(q, n_equil + (q + 1) * stride - 1) for q in range(first, first + 3 * n)]
    for h in range(3):
        at, _ = pmf.pmf_od1d_records(h, n_equil, stride, start, n)
        assert np.all(at % 3 == h)

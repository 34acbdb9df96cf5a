"""The bench's bytes of a V-cycle applied as a preconditioner: what that kernel
moves, without the FP64 residual and update of a solve."""
import pytest

import bench


def test_preconditioner_bytes():
    # FP32, 3D, 3+3 sweeps, per fine cell and phase.  Sweeps: read x and b, write x, read the flag byte, 13 B each;
    # the first pass of the first one starts from zero and reads no x (2 B less: 4 B of half the cells).
    # Residual + restriction: x 4, red b 2, red flags 1/2, per coarse cell b 4 + flags 1; prolongation: x read
    # and written 8, flags 1, per coarse cell x 4.  Level sum 8/7.
    v = (6 * 13 - 2) + (4 + 2 + 0.5 + 5 / 8) + (8 + 1 + 4 / 8)
    assert bench.split_vcycle_bytes(3, 4, 6) == pytest.approx(v * 8 / 7)
    # around it: b read in FP64 (8 B), level 0's b written (4) and its flags read (1); its x read (4) with the
    # flags (1) and the result read and written in FP64 (16)
    assert bench.precond_bytes(1000, 3, True, 5, sweeps=6) == pytest.approx(5 * 1000 * (v * 8 / 7 + 34))
    # FP64, 2D, 2+2 sweeps
    v = (4 * 25 - 4) + (8 + 4 + 0.5 + 9 / 4) + (16 + 1 + 8 / 4)
    assert bench.split_vcycle_bytes(2, 8, 4) == pytest.approx(v * 4 / 3)
    assert bench.precond_bytes(10, 2, False, 1, sweeps=4) == pytest.approx(10 * (v * 4 / 3 + 8 + 8 + 1 + 8 + 1 + 16))

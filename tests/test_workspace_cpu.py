"""Device memory of a driver (gp_workspace_size, no GPU needed)."""
import ctypes

import pytest

from paper_2604_16613_gb300 import circuits as C
from paper_2604_16613_gb300 import native
from paper_2604_16613_gb300.dem import Bounds

NM = C.NoiseModel.uniform(1e-3)


def workspace(bounds):
    cb, size = bounds.to_c(), ctypes.c_uint64()
    native.check(native.load().gp_workspace_size(ctypes.byref(cb), ctypes.byref(size)))
    return size.value


@pytest.mark.parametrize("make,limit_mb", [
    # what these drivers took while stage 1 still left one 16-byte record per
    # mechanism and word (measured): a plane record per noise row takes no more
    (lambda: [C.rotated_surface_code_memory(3, 3, NM)], 69.1),
    (lambda: [C.rotated_surface_code_memory(11, 11, NM)], 104.8),
    (lambda: [C.rotated_surface_code_memory(25, 25, NM)], 470.2),
    (lambda: [C.rotated_surface_code_memory(45, 9, NM)], 597.4),
    (lambda: [C.bb_memory(12, NM, seed=3)], 162.8),
    (lambda: [C.repetition_code_memory(25, 100, NM)], 102.3),
    (lambda: C.adaptive_branches(n=16, d=10, lo=10, hi=30, seed=4, noise=NM), 4823.0),
    (lambda: [C.rotated_surface_code_memory(3 + i % 5, 2 + (i * 5) % 7, NM) for i in range(64)], 271.1),
], ids=["surface3", "surface11", "surface25", "surface45", "bb12", "repetition25x100", "adaptive16", "small_batch"])
def test_workspace_bytes(make, limit_mb):
    assert workspace(Bounds.for_circuits(make())) <= limit_mb * 1e6

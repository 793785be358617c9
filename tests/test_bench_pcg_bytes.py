"""Bytes the PCG roofline divides by: the iteration of the pass chain does not
store A p, the plain-form baseline does."""
import os
import sys

sys.path.insert(0, os.path.join(os.path.dirname(__file__), ".."))
import bench  # noqa: E402


def test_pcg_iteration_bytes_of_the_fused_chain():
    c = 8
    passes_1_to_4 = (3 + 6) * c + 12 * c + (12 * c + 4) + 12 * c
    divergence_and_residual = 6 * c + 3 * c + 3 * c       # stresses in, r in and out
    directions = 9 * c + 6 * c                            # r, p, x in; p, x out
    for variant in (0, 1):
        assert bench.pcg_bytes_per_voxel(variant) == passes_1_to_4 + divergence_and_residual + directions
    assert bench.pcg_bytes_per_voxel(2) == 54 * c + 4 + (9 + 15) * c

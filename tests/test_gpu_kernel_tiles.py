"""Kernel generation in tiles of 8 rows (meshes of few tiles) and of 16 rows
gives the same kernel at the same offsets.  Bar: two evaluations of the same
corner terms differ by roundings of the terms, 2e-15 of the eight corners'
magnitudes; those are at most 8 for the second derivatives (asinh of ratios
below 1000, arc tangents) and 8 times the coordinates' sum for the first."""
import pytest
import torch

from paper_2005_10160_gb300 import capi
from paper_2005_10160_gb300.plan import kernel_values

pytestmark = pytest.mark.gpu

CELL = (20.0, 25.0, 15.0, 8.0)


@pytest.mark.parametrize("comps", [0x7F, 0x3F | capi.GRAV_GX | capi.GRAV_GY])
@pytest.mark.parametrize("size", [(33, 17, 3), (40, 8, 3), (5, 31, 3), (1, 1, 3)])
def test_tiles_of_8_and_16_rows_agree(gravlib, size, comps):
    nx, ny, nz = size
    big = kernel_values((320, 260, nz, *CELL), comps)
    big = big[:, :, 260 - ny:259 + ny, 320 - nx:319 + nx]
    got = kernel_values((*size, *CELL), comps)
    reach = (nx + 1) * 20.0 + (ny + 1) * 25.0 + 8.0 + (nz + 1) * 15.0
    for slot, c in enumerate(capi.comp_list(comps)):
        bar = 2e-15 * 6.672e-11 * 8 * 8 * (reach if c in (0, 7, 8) else 1.0)
        assert float((got[slot] - big[slot]).abs().max()) <= bar, c
        assert float(big[slot].abs().max()) > 1e3 * bar or size == (1, 1, 3)

"""FP32 storage adds its partial sums with at least FP64's 53 bits.

Sums whose large terms cancel exactly: 1 + y + 2^-51 - 1 - y with y just below
2^-24. FP64 holds every running sum exactly (1 + y ends at 2^-45, its last bit
for sums near 1 is 2^-52), and so do the FP32 products that are summed, so the
result is 2^-51 to the last bit. Two floats lose it: next to y, the last bit
of the second one is 2^-48.
"""
import numpy as np
import pytest

from gpu_common import context, water

pytestmark = pytest.mark.gpu

Y = 2.0 ** -25 * (2.0 - 2.0 ** -20)   # 21 bits: as TF32 parts too it is exact
TERMS = np.array([1.0, Y, 2.0 ** -51, -1.0, -Y])


def test_transform_adds_its_partial_sums_in_fp64():
    """F_ij = sum_r C[r, i] (X C)[r, j] with X = 1 and one term in each of five rounds of 32 row blocks."""
    s = water(160)
    ctx = context(s, precision=1)
    ctx.set_thresholds(1e-20, 1e-3, 1e-8)
    mn = ctx.get_blocks()[0]
    X = np.zeros((len(mn), 6, 6))
    X[mn[:, 0] == mn[:, 1]] = np.eye(6)
    n_occ_tiles = int(sum(-(-4 * k // 16) for k in np.bincount(s.group_of_mol)))
    nt = np.full(s.n_mol, 2, dtype=np.int32)
    tiles = np.tile([0, n_occ_tiles], s.n_mol).astype(np.int32)   # group 0's first occupied and virtual tile
    vals = np.zeros((s.n_mol, 2, 6, 16))
    vals[::32, 0, 0, 0] = 1.0
    vals[::32, 1, 0, 0] = TERMS
    ctx.set_C_tiles(nt, tiles, vals.reshape(-1, 6, 16))
    ctx.set_fock_blocks(X)
    ctx.rotate_sweep()
    F_ov, _ = ctx.get_F()
    ctx.close()
    assert F_ov[0, 0] == 2.0 ** -51

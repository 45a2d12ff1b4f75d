"""FP32 storage adds its partial sums with at least FP64's 53 bits.

Sums whose large terms cancel exactly: 1 + y + 2^-51 - 1 - y with y just below
2^-24. FP64 holds every running sum exactly (1 + y ends at 2^-45, its last bit
for sums near 1 is 2^-52), and so do the FP32 products that are summed, so the
result is 2^-51 to the last bit. Two floats lose it: next to y, the last bit
of the second one is 2^-48.
"""
import numpy as np
import pytest

from gpu_common import P, context, water

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


def test_gradients_add_their_products_in_fp64():
    """dE/dV0 (ss-sigma) of two molecules that share ten occupied tiles, one term of P in every second one:
    both ordered pairs of the O s orbitals, P = 2 sum, times the decay at their distance (a square root,
    a division and an exponential of about -4, a few units in the last place each)."""
    s = water(40)
    ctx = context(s, precision=1)
    n_tiles = int(sum(-(-4 * k // 16) for k in np.bincount(s.group_of_mol)))
    assert n_tiles >= 10
    nt = np.zeros(s.n_mol, dtype=np.int32)
    nt[:2] = 10
    vals = np.zeros((2, 10, 6, 16))
    vals[0, ::2, 0, 0] = 1.0
    vals[1, ::2, 0, 0] = TERMS
    ctx.set_C_tiles(nt, np.tile(np.arange(10, dtype=np.int32), 2), vals.reshape(-1, 6, 16))
    _, dpar = ctx.gradients()
    ctx.close()
    O = s.xyz.reshape(-1, 3, 3)[:2, 0]
    r = np.sqrt(((O[1] - O[0]) ** 2).sum())
    assert r < P["r_cut"]
    ref = 2.0 * 2.0 * 2.0 ** -51 * np.exp(-r / P["r_decay"])
    assert abs(dpar[0] - ref) <= 64 * 2.0 ** -53 * ref

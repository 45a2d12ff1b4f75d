"""The adjoint where the molecules of a group hold different tiles.

Random occupied MOs of which every row block holds some tiles and lacks others
(down to one tile, one row none at all). With every pair of groups neighbours
W = 2 C_o F_oo C_o^T equals the oracle's 1/2 P H P for any MOs, as in the test on
ragged groups, with its tolerances: FP64 1e-9 of the largest component, FP32
storage 2e-5.
"""
import numpy as np
import pytest

from gpu_common import P, library, water
from oracle import adjoint

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[8, 7, 3], [4, 8, 6], [2, 1, 5, 8, 8]])
@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 2e-5)])
def test_gradients_of_rows_with_absent_tiles(sizes, prec, tol):
    library()
    from paper_1402_2880_gb300 import Context
    rng = np.random.default_rng(sum(sizes) + prec)
    s = water(sum(sizes), seed=6, sigma=0.05)
    groups = np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)
    ctx = Context(s.species, s.xyz, groups, P, precision=prec)
    assert (ctx.colouring() >= 0).all()
    mos = np.concatenate([np.minimum(16, 4 * k - np.arange(0, 4 * k, 16)) for k in sizes])   # MOs of every tile
    nt, tiles, vals = [], [], []
    for r in range(s.n_mol):
        t = np.nonzero(rng.random(mos.size) < (0.0, 0.3, 0.6)[min(r, 1 + r % 2)])[0]
        if r == 1:
            t = t[:1]
        nt.append(t.size)
        tiles.append(t)
        v = rng.normal(0.0, 0.2, (t.size, 6, 16)).astype(np.float32)
        vals.append(v * (np.arange(16) < mos[t][:, None])[:, None, :])
    ctx.set_C_tiles(np.array(nt), np.concatenate(tiles), np.concatenate(vals))
    g, gp = ctx.gradients()
    Co = ctx.get_C()[:, :ctx.n_occ]
    _, dq, _ = ctx.get_charges()
    ctx.close()
    assert np.count_nonzero(Co) > 0
    rg, rgp = adjoint.gradients(s, P, 2.0 * Co @ Co.T, dq)
    assert np.abs(g - rg).max() <= tol * np.abs(rg).max()
    assert np.abs(gp - rgp).max() <= tol * np.abs(rgp).max()

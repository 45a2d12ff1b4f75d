"""The pair selection in one CTA and in launches picks the same rotations.

A single cluster of up to 64 blocks (8 x 8 groups, all neighbours) takes one CTA, larger
ones and clusters of a batch the launches: each cluster of a batch of two selects
exactly the pairs that it selects alone, on both sides of that line, without and with
more candidates than the cap.
"""
import numpy as np
import pytest

from gpu_common import P, library, water
from synth import concat_clusters

pytestmark = pytest.mark.gpu


def _pairs(s, prec, factor):
    from paper_1402_2880_gb300 import Context
    ctx = Context.from_system(s, dict(P, rot_cap_factor=factor), precision=prec)
    ctx.set_thresholds(1e-4, 1e-3, 1e-8)
    ctx.guess()
    ctx.orthonormalise(0, max_pass=5)
    ctx.build_fock()
    n, _ = ctx.rotate_sweep()
    _, _, i, j = ctx.pairs()
    n_occ, n_blk = ctx.n_occ, int((ctx.colouring() >= 0).sum())
    ctx.close()
    assert n == i.size
    return set(zip(i.tolist(), (j - n_occ).tolist())), n_blk


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("factor", [0.5, 10.0])
@pytest.mark.parametrize("n,one_cta", [(27, True), (64, True), (80, False)])
def test_one_cta_and_launches_select_the_same_pairs(n, one_cta, factor, prec):
    library()
    a, b = water(n, seed=3), water(8, seed=4)
    alone, n_blk = _pairs(a, prec, factor)
    assert (n_blk <= 64) == one_cta
    assert _pairs(a, prec, factor)[0] == alone
    other, _ = _pairs(b, prec, factor)
    both, _ = _pairs(concat_clusters([a, b]), prec, factor)
    shifted = {(i + 4 * a.n_mol, j + 2 * a.n_mol) for i, j in other}
    assert alone and both == alone | shifted

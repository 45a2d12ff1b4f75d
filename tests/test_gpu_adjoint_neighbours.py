"""The adjoint on more neighbouring groups than one launch takes.

140 groups of one molecule, all of them neighbours of each other (as in the
ragged-groups test, W then equals the oracle's 1/2 P H P): a group's 140
neighbours are taken 128 and 12. Tolerances as there: FP64 to 1e-9 of the largest
component, FP32 storage to 2e-5.
"""
import numpy as np
import pytest

from gpu_common import P, library, water
from oracle import adjoint

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 2e-5)])
def test_gradients_with_more_neighbours_than_a_lookup(prec, tol):
    library()
    from paper_1402_2880_gb300 import Context
    n = 140
    s = water(n, seed=4, sigma=0.05)
    p = dict(P, group_cut=200.0)
    ctx = Context(s.species, s.xyz, np.arange(n, dtype=np.int32), p, precision=prec)
    assert (ctx.colouring() >= 0).all()
    ctx.set_thresholds(1e-4, 1e-3, 1e-8)
    ctx.guess()
    ctx.orthonormalise(0, max_pass=5)
    g, gp = ctx.gradients()
    Co = ctx.get_C()[:, :ctx.n_occ]
    _, dq, _ = ctx.get_charges()
    ctx.close()
    rg, rgp = adjoint.gradients(s, p, 2.0 * Co @ Co.T, dq)
    assert np.abs(g - rg).max() <= tol * np.abs(rg).max()
    assert np.abs(gp - rgp).max() <= tol * np.abs(rgp).max()


def test_gradients_with_a_group_that_neighbours_all():
    """One group of eight molecules spread over a 14 x 14 x 14 lattice of single-molecule groups has 2737
    neighbours, more than fit shared memory at once. The guess's MOs in both precisions: FP32 rounds
    them, F and Z, as above 2e-5."""
    library()
    import torch
    from paper_1402_2880_gb300 import Context
    if torch.cuda.mem_get_info()[0] < 150 * 2 ** 30:
        pytest.skip("the pair lists of 1.7 million neighbours take 100 GB")
    s = water(14 ** 3)
    O = s.xyz.reshape(-1, 3, 3)[:, 0]
    site = np.rint((O - O.min(0)) / (3.1 / 0.529177)).astype(int)
    hub = np.isin(site, (3, 10)).all(1)
    assert hub.sum() == 8
    groups = np.zeros(s.n_mol, dtype=np.int32)
    groups[~hub] = np.arange(1, s.n_mol - 7)
    out = []
    for prec in (0, 1):
        ctx = Context(s.species, s.xyz, groups, dict(P, group_cut=36.0), precision=prec)
        assert (ctx.colouring()[0] >= 0).all()
        ctx.guess()
        out.append(ctx.gradients())
        ctx.close()
    for a, b in zip(*out):
        assert np.abs(a).max() > 0 and np.abs(a - b).max() <= 2e-5 * np.abs(a).max()

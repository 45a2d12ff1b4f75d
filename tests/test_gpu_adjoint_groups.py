"""The adjoint on groups of 1 to 8 molecules, in both storage precisions, against the oracle.

With every pair of groups neighbours, W = 2 C_o F_oo C_o^T equals the oracle's 1/2 P H P for any
occupied MOs, so the gradients of the oracle (fed the GPU's own MOs) are those of the GPU up to
rounding: FP64 to 1e-9 of the largest component, FP32 storage (MOs, F_oo and Z rounded to FP32,
sums of a few hundred terms) to 2e-5.
"""
import numpy as np
import pytest

from gpu_common import P, library, water
from oracle import adjoint

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[1], [1, 2, 3, 4, 5, 3], [8, 7, 3], [4, 8, 6]])
@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 2e-5)])
def test_gradients_on_ragged_groups(sizes, prec, tol):
    library()
    from paper_1402_2880_gb300 import Context
    s = water(sum(sizes), seed=4, sigma=0.05)
    groups = np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)
    ctx = Context(s.species, s.xyz, groups, P, precision=prec)
    assert (ctx.colouring() >= 0).all()
    ctx.set_thresholds(1e-4, 1e-3, 1e-8)
    ctx.guess()
    ctx.orthonormalise(0)
    g, gp = ctx.gradients()
    Co = ctx.get_C()[:, :ctx.n_occ]
    _, dq, _ = ctx.get_charges()
    rg, rgp = adjoint.gradients(s, P, 2.0 * Co @ Co.T, dq)
    assert np.abs(g - rg).max() <= tol * np.abs(rg).max()
    assert np.abs(gp - rgp).max() <= tol * np.abs(rgp).max()

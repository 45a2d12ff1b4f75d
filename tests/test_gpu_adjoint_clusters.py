"""Gradients of several clusters in one context are those of each cluster.

Nothing couples two clusters, so the forces are the clusters' own and the parameter
gradients their sum. In FP64 they equal those of each cluster alone: only the
order of FP64 additions differs (the shares of the gamma forces follow the largest
cluster; the parameters are summed over all molecules), a few hundred of them, 1e-12
of the largest component. In mixed precision gamma's FP32 partial sums are taken
over other atoms, so each cluster is compared with the oracle instead, with the
tolerances of the ragged-groups test (every pair of groups of a cluster neighbours;
FP64 1e-9 of the largest component, FP32 storage 2e-5).
"""
import numpy as np
import pytest

from gpu_common import P, context, water
from oracle import adjoint
from synth import concat_clusters

pytestmark = pytest.mark.gpu


def _prepared(s, prec):
    ctx = context(s, precision=prec)
    ctx.set_thresholds(1e-4, 1e-3, 1e-8)
    ctx.guess()
    ctx.orthonormalise(0, max_pass=3)
    return ctx


@pytest.mark.parametrize("sizes", [(13, 50), (1, 27, 8, 125)])
def test_fp64_gradients_of_a_batch_equal_each_cluster_alone(sizes):
    parts = [water(n, seed=k) for k, n in enumerate(sizes)]
    g, gp = _prepared(concat_clusters(parts), 0).gradients()
    alone = [_prepared(p, 0).gradients() for p in parts]
    ref, refp = np.concatenate([a[0] for a in alone]), [a[1] for a in alone]
    assert np.abs(g - ref).max() <= 1e-12 * np.abs(ref).max()
    assert np.abs(gp - sum(refp)).max() <= 1e-12 * sum(np.abs(r) for r in refp).max()


@pytest.mark.parametrize("sizes", [(3, 20), (17, 1, 8, 25)])
@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 2e-5)])
def test_gradients_of_a_batch_match_the_oracle(sizes, prec, tol):
    parts = [water(n, seed=k + 3, sigma=0.05) for k, n in enumerate(sizes)]
    ctx = _prepared(concat_clusters(parts), prec)
    g, gp = ctx.gradients()
    Co = ctx.get_C()[:, :ctx.n_occ]
    _, dq, _ = ctx.get_charges()
    col = ctx.colouring()
    ctx.close()
    m0 = g0 = 0
    refp = 0.0
    for s in parts:
        at = slice(3 * m0, 3 * (m0 + s.n_mol))
        C = Co[6 * m0:6 * (m0 + s.n_mol)]
        assert (col[g0:g0 + s.n_groups, g0:g0 + s.n_groups] >= 0).all()
        rg, rgp = adjoint.gradients(s, P, 2.0 * C @ C.T, dq[at])
        assert np.abs(g[at] - rg).max() <= tol * np.abs(rg).max()
        refp = refp + rgp
        m0 += s.n_mol
        g0 += s.n_groups
    assert np.abs(gp - refp).max() <= tol * np.abs(refp).max()

"""The guess resolves eigenvalues that nearly coincide.

Equal on-site energies and S = 1 with couplings of relative size `scale`: all six
eigenvalues of a molecule lie within it. The eigenvectors have to be accurate to
the rounding of the matrix all the same: |H x - (x^T H x) x| is that of a
backward-stable eigensolver (Jacobi: a few units per sweep, 64 u = 7e-15 of |H|
here), not the size of the couplings.
"""
import numpy as np
import pytest

from gpu_common import P, library, water

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-3, 1e-11, 1e-12, 1e-13, 1e-14])
def test_guess_of_a_nearly_degenerate_molecule(scale):
    library()
    from paper_1402_2880_gb300 import Context
    p = dict(P, onsite_O_s=-0.5, onsite_O_p=-0.5, onsite_H_s=-0.5, S0=[0.0] * 4,
             V0=[scale * v for v in P["V0"]])
    s = water(8)
    ctx = Context.from_system(s, p, precision=0)
    ctx.set_thresholds(1e-6, 1e-5, 1e-8)
    ctx.guess()
    C = ctx.get_C()
    mn, _, H0, _ = ctx.get_blocks()
    for H, m in zip(H0[mn[:, 0] == mn[:, 1]], mn[mn[:, 0] == mn[:, 1]][:, 0]):
        rows = C[6 * m:6 * m + 6]
        x = rows[:, np.abs(rows).max(0) > 0].astype(np.longdouble)
        assert x.shape == (6, 6)
        assert np.abs(x.T @ x - np.eye(6)).max() <= 64 * 2.0 ** -53
        lam = np.einsum("ki,kl,li->i", x, H.astype(np.longdouble), x)
        res = np.sqrt(((H @ x - x * lam) ** 2).sum(0).astype(float))
        assert res.max() <= 64 * 2.0 ** -53 * np.linalg.norm(H)
    ctx.close()

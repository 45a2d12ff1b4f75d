"""The FP32 transform, overlap transform and density at sizes that leave their units partly filled.

Systems of 1 to 65 molecules (tiles with fewer rows than one round takes, a
last round of 1 to 3 row blocks, pairs of one partial sum and of several),
against FP64 products of the same FP32 MOs:

* F = C^T H C within 1024 u times the sum of the absolute terms (u = 2^-24; the
  bound of the larger sizes: H, Y = H C and F rounded once each, a value of Y
  sums 6 terms per neighbour, F at most 192 terms between flushes);
* P = 2 C_occ C_occ^T within 36 u times the sum of the absolute terms: FP32
  sums of at most 32 products (one rounding each), added up without a rounding
  that matters, 2 sums of half the tiles, and a few units spare.
"""
import numpy as np
import pytest

from gpu_common import context, oracle_scf, water
from oracle import sparse

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.mark.parametrize("n", [1, 2, 5, 17, 33, 65])
def test_fp32_transform_and_density(n):
    eps = 1e-6
    s, sc = water(n), oracle_scf(n)
    ctx = context(s, precision=1)
    ctx.set_thresholds(eps, 10 * eps, 1e-8)
    ctx.guess()
    ctx.orthonormalise(0)
    C0 = ctx.get_C()
    Q = np.random.default_rng(n).normal(0.0, 0.05, s.n_atoms)
    ctx.set_charges(Q_in=Q)
    ctx.build_fock()
    ctx.rotate_sweep()
    F, Fd = ctx.get_F()
    H = sparse.fock(sc.H0, sc.S, Q, sc.atom_of_ao, eps)
    F_ref, Fd_ref, mask = sparse.transform_ov(C0, H, sc.st)
    terms = np.abs(C0).T @ (np.abs(H) @ np.abs(C0))
    no = sc.st.n_occ
    assert np.all(np.abs(F - F_ref) <= 1024 * U * np.where(mask, terms[:no, no:], 0.0))
    assert np.all(np.abs(Fd - Fd_ref) <= 1024 * U * np.diag(terms))
    Co = ctx.get_C()[:, :no]
    Pref, Pabs = 2.0 * Co @ Co.T, 2.0 * np.abs(Co) @ np.abs(Co).T
    mn = ctx.get_blocks()[0]
    for (m, k), blk in zip(mn, ctx.density_blocks()):
        at = np.ix_(range(6 * m, 6 * m + 6), range(6 * k, 6 * k + 6))
        assert np.all(np.abs(blk - Pref[at]) <= 36 * U * Pabs[at])
    ctx.close()


@pytest.mark.parametrize("n", [1, 5, 33, 65])
def test_fp32_overlaps(n):
    s, sc = water(n), oracle_scf(n)
    ctx = context(s, precision=1)
    ctx.set_thresholds(1e-6, 1e-5, 1e-8)
    ctx.guess()
    ctx.orthonormalise(0)
    C0 = ctx.get_C()
    ctx.orthonormalise(1, max_pass=1)
    sigma = ctx.get_overlap()
    no = sc.st.n_occ
    mos = np.arange(no)
    mask = sparse.overlap_mask(sc.st, mos)
    ref = np.where(mask, C0[:, mos].T @ (sc.S @ C0[:, mos]), 0.0)
    terms = np.abs(C0[:, mos]).T @ (np.abs(sc.S) @ np.abs(C0[:, mos]))
    assert np.all(np.abs(sigma - ref) <= 1024 * U * np.where(mask, terms, 0.0))
    ctx.close()

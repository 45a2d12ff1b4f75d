"""Grouping at the edges of the matching kernel's ranges, bit for bit against the oracle: one
molecule, one molecule per centre, the last size of one CTA with its lists in shared memory and the
first of many CTAs with them in global memory, and more centres than one CTA's shared memory lists
(those lists are in global memory, written by many CTAs)."""
import numpy as np
import pytest

from gpu_common import library
from oracle import kmeans
from synth import lattice_water

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_link,max_iter", [(1, 8, 100), (7, 1, 100), (130, 3, 0), (512, 7, 3), (513, 7, 3),
                                               (2001, 1, 2)])
def test_groups_match_oracle(n, n_link, max_iter):
    library()
    from paper_1402_2880_gb300 import group_molecules
    s = lattice_water(n, seed=3, displace_sigma_A=0.4)
    g, ng, it = group_molecules(s.xyz, n_link=n_link, max_iter=max_iter)
    rg, rng_, rit = kmeans.group_molecules(s.xyz, n_link=n_link, max_iter=max_iter)
    assert (ng, it) == (rng_, rit)
    assert np.array_equal(g, rg)

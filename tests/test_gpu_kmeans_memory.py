"""The grouping without room for the table of distances gives the same groups.

The table is optional: an allocator that refuses it (it is the largest buffer by far)
leaves the matching to compute distances as it goes, with one CTA (lists in shared
memory) and with many. Nothing is left allocated, and a refusal of any other buffer is
SSCF_ERR_OOM.
"""
import ctypes

import numpy as np
import pytest

from gpu_common import library, water

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_link", [(343, 8), (343, 1), (1000, 7)])
def test_grouping_without_the_distance_table(n, n_link):
    lib = library()
    import torch
    from paper_1402_2880_gb300 import _lib
    xyz = water(n, sigma=0.5).xyz
    ref = _lib.group_molecules(xyz, n_link=n_link)
    live, refused, sizes, limit = {}, [], [], [8 * n * (n // n_link)]   # the table has at least that many bytes

    def alloc(n_bytes, _user):
        if n_bytes >= limit[0]:
            refused.append(n_bytes)
            return None
        sizes.append(n_bytes)
        t = torch.empty(n_bytes, dtype=torch.uint8, device="cuda")
        live[t.data_ptr()] = t
        return t.data_ptr()

    def release(ptr, _user):
        live.pop(ptr)
    hooks = _lib.ALLOC_FN(alloc), _lib.FREE_FN(release)
    assert lib.sscf_set_allocator(*hooks, None) == 0
    try:
        got = _lib.group_molecules(xyz, n_link=n_link)
        assert len(refused) == 1 and not live
        limit[0] = max(sizes)
        with pytest.raises(_lib.SscfError) as e:
            _lib.group_molecules(xyz, n_link=n_link)
        assert e.value.status == -2 and not live
    finally:
        assert lib.sscf_set_allocator(ctypes.cast(None, _lib.ALLOC_FN), ctypes.cast(None, _lib.FREE_FN), None) == 0
    assert np.array_equal(got[0], ref[0]) and got[1:] == ref[1:]

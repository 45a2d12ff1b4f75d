"""The adjoint's working memory: allocated by the first gradients call, not at creation.

A refusing allocator at that call gives SSCF_ERR_OOM with the context unchanged,
also when only the second of the two buffers is refused; the next call gets what is
missing and gives the result of an undisturbed context.
"""
import ctypes

import numpy as np
import pytest

from gpu_common import context, library, water

pytestmark = pytest.mark.gpu


def test_first_gradients_call_allocates_and_survives_refusals():
    lib = library()
    import torch
    from paper_1402_2880_gb300 import _lib
    live, allowed = {}, [10 ** 9]

    def alloc(n_bytes, _user):
        if allowed[0] <= 0:
            return None
        allowed[0] -= 1
        t = torch.empty(n_bytes, dtype=torch.uint8, device="cuda")
        live[t.data_ptr()] = t
        return t.data_ptr()

    def release(ptr, _user):
        live.pop(ptr)
    s = water(27)
    ref_ctx = context(s)
    ref_ctx.guess()
    ref = ref_ctx.gradients()
    ref_ctx.close()
    hooks = _lib.ALLOC_FN(alloc), _lib.FREE_FN(release)
    assert lib.sscf_set_allocator(*hooks, None) == 0
    try:
        ctx = context(s)
        ctx.guess()
        for refusal in (0, 1):
            allowed[0] = refusal
            q = ctx.get_charges()
            with pytest.raises(_lib.SscfError) as e:
                ctx.gradients()
            assert e.value.status == -2
            assert all(np.array_equal(a, b) for a, b in zip(q, ctx.get_charges()))
        allowed[0] = 1   # the first buffer is there, the second is missing
        got = ctx.gradients()
        allowed[0] = 0   # both are kept
        again = ctx.gradients()
        ctx.close()
        assert not live
    finally:
        assert lib.sscf_set_allocator(ctypes.cast(None, _lib.ALLOC_FN), ctypes.cast(None, _lib.FREE_FN), None) == 0
    for a, b, r in zip(got, again, ref):
        assert np.array_equal(a, r) and np.array_equal(b, r)

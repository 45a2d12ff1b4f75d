"""The FP32 sweep kernel on partly filled groups equals the generic kernel bit for bit.

Groups of every size from 1 to 8 molecules (so every modulus of the in-block
colour, in passes over all MOs and over the occupied ones) with row counts that
leave last runs and flag words partly filled; with one closure per sweep and
with one per colour. The two kernels apply the same FP32 updates in the same
order, so C and the tile structure agree exactly.
"""
import numpy as np
import pytest

from gpu_common import P, library, water

pytestmark = pytest.mark.gpu


def _groups(n, kind):
    if kind == "ramp":      # 1, 2, ..., 8, 1, 2, ... molecules
        sizes = np.tile(np.arange(1, 9), n // 36 + 1)
    elif kind == "sevens":  # odd, no full group
        sizes = np.full(n, 7)
    else:                   # full groups and one small rest
        sizes = np.full(n, 8)
    return np.repeat(np.arange(sizes.size), sizes)[:n].astype(np.int32)


@pytest.mark.parametrize("n,kind,closure", [(1, "ramp", 0), (37, "ramp", 0), (97, "ramp", 0), (131, "sevens", 0),
                                            (129, "eights", 0), (97, "ramp", 1)])
def test_sweeps_of_partly_filled_groups_match_the_generic_kernel(n, kind, closure):
    library()
    from paper_1402_2880_gb300 import Context
    s = water(n)
    out = []
    for variant in (0, 1):
        ctx = Context(s.species, s.xyz, _groups(n, kind), P, precision=1, apply_variant=variant, closure_mode=closure)
        ctx.set_thresholds(1e-3, 1e-2, 1e-8)
        ctx.guess()
        ctx.orthonormalise(0, max_pass=20)
        ctx.set_thresholds(1e-5, 1e-4, 1e-6)
        ctx.reset_charges()
        infos = [ctx.step() for _ in range(2)]
        out.append((ctx.get_C_tiles(), infos))
        ctx.close()
    (nt0, t0, v0), i0 = out[0]
    (nt1, t1, v1), i1 = out[1]
    assert np.array_equal(nt0, nt1) and np.array_equal(t0, t1)
    assert np.array_equal(v0, v1)
    for a, b in zip(i0, i1):
        for k in ("energy", "n_rot", "n_combo", "upd_rot", "upd_combo", "eta"):
            assert a[k] == b[k], k


@pytest.mark.parametrize("n,kind", [(1, "ramp"), (37, "ramp"), (97, "ramp"), (131, "sevens")])
def test_fp64_sweeps_match_the_generic_kernel(n, kind):
    """FP64 storage: one sweep and one pass of each kind. The products of a rotation may be
    contracted differently (an ulp of 1 per update, 200 updates of a value at most: 1e-13)."""
    library()
    from paper_1402_2880_gb300 import Context
    s = water(n)
    out = []
    for variant in (0, 1):
        ctx = Context(s.species, s.xyz, _groups(n, kind), P, precision=0, apply_variant=variant)
        ctx.set_thresholds(1e-4, 1e-3, 1e-8)
        ctx.guess()
        ctx.orthonormalise(0, max_pass=1)
        ctx.orthonormalise(1, max_pass=1)
        ctx.build_fock()
        ctx.rotate_sweep()
        out.append(ctx.get_C())
        ctx.close()
    assert np.abs(out[0] - out[1]).max() <= 1e-13

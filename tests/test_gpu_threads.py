"""Calls of different sizes from several host threads at the same time.

Contexts are independent and so are groupings: a kernel's launch limits, which
belong to the kernel, must not depend on the sizes of whoever set them last.
"""
import threading

import numpy as np
import pytest

from gpu_common import context, library, water

pytestmark = pytest.mark.gpu


def _together(*jobs):
    errors = []
    start = threading.Barrier(len(jobs))

    def run(job):
        try:
            start.wait()
            job()
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(e)
    threads = [threading.Thread(target=run, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert errors == []


def test_groupings_of_different_sizes():
    library()
    from paper_1402_2880_gb300._lib import group_molecules
    sizes = [(8, 4), (512, 1)]   # lists of a few hundred bytes and of 56 KB
    xyz = [water(n, sigma=0.5).xyz for n, _ in sizes]
    alone = [group_molecules(x, n_link=k)[0] for x, (_, k) in zip(xyz, sizes)]

    def job(i, times):
        def run():
            for _ in range(times):
                assert np.array_equal(group_molecules(xyz[i], n_link=sizes[i][1])[0], alone[i])
        return run
    _together(job(0, 400), job(1, 40))


@pytest.mark.parametrize("precision", [0, 1])
def test_steps_and_gradients_of_contexts_of_different_sizes(precision):
    import torch
    sizes = (8, 300)
    streams = [torch.cuda.Stream() for _ in sizes]
    ctxs = [context(water(n), precision=precision, stream=s.cuda_stream) for n, s in zip(sizes, streams)]
    for c in ctxs:
        c.set_thresholds(1e-3, 1e-2, 1e-8)
        c.guess()

    def job(c, times):
        def run():
            for _ in range(times):
                c.guess()
                c.orthonormalise(0, max_pass=2)
                c.step()
                c.gradients()
        return run
    _together(job(ctxs[0], 120), job(ctxs[1], 20))
    for c in ctxs:
        c.close()

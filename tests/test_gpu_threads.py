"""Host threads that step different contexts at the same time, each on its own stream.

A context belongs to one thread at a time; different contexts share nothing that a step changes, whichever kernel
instance they run.  Contexts of one size with different shared-memory needs (material tables, currents and probes, ring
depths) run the same instance, so their launches meet at its launch limits; every thread's fields equal the same steps
taken alone.
"""
import threading

import numpy as np
import pytest

import cavity_inputs as ci
from tests.gpu_util import DT

pytestmark = pytest.mark.gpu


def _media(dims, count):
    """count materials (scaled vacuum) in layers along z."""
    if count == 0:
        return None, None
    nx, ny, nz = dims
    eps = 1.0 + (np.arange(nz + 1) % count) / 8.0
    ce = np.broadcast_to((DT / eps)[:, None, None], (nz + 1, ny + 1, nx + 1)).astype(np.float32)
    return [np.ascontiguousarray(ce)] * 3, None


def _solve(dims, job, calls, stream=None, start=None):
    from paper_2504_09118_gb300 import Cavity
    tuning, materials, probes = job
    ce, ch = _media(dims, materials)
    with Cavity(*dims, DT, 1.0, ce, ch, 0, stream) as cav:
        cav.tune(**tuning)
        cav.set_fields(ci.random_fields(51, *dims))
        if probes:
            cav.set_probes([(q % 6, q % dims[0], q % dims[1], q % dims[2]) for q in range(probes)], 8)
        if start:
            start.wait()
        for n in calls:
            cav.step(n)
        return cav.get_fields()


ON_CHIP = [({}, 0, 0), ({}, 20, 0), ({}, 0, 200), ({}, 20, 100)]
RINGS = [(dict(kernel=3, tile_y=12, stages=s), 0, 0) for s in (3, 6, 4, 5)]


@pytest.mark.parametrize("jobs,dims,calls", [(ON_CHIP, (40, 33, 21), [4] * 600), (RINGS, (64, 33, 29), [200] * 40)],
                         ids=["on chip", "ring depths"])
def test_threads_with_different_launch_needs(jobs, dims, calls):
    import torch
    want = [_solve(dims, j, calls) for j in jobs]
    streams = [torch.cuda.Stream() for _ in jobs]
    start = threading.Barrier(len(jobs))
    got, errors = [None] * len(jobs), []

    def work(n):
        try:
            got[n] = _solve(dims, jobs[n], calls, streams[n], start)
        except Exception as e:   # reported by the test's own thread
            errors.append((n, e))
            start.abort()

    threads = [threading.Thread(target=work, args=(n,)) for n in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for a, b in zip(got, want):
        for x, y in zip(a, b):
            np.testing.assert_array_equal(x, y)

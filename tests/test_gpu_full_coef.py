"""Per-position coefficient arrays (more than 256 distinct tuples) under AUTO and TEMPORAL: two steps per launch,
the coefficients streamed with the fields.  FP32 results equal the unfused kernel's bit for bit (same operations);
16-bit storage rounds once per two steps, so against FP32 its error is a random walk of half as many roundings,
bounded as elsewhere by 3 (u / sqrt 3) sqrt(N + 1)."""
import math

import numpy as np
import pytest

import cavity_inputs as ci
from tests.gpu_util import DT

pytestmark = pytest.mark.gpu

# around the 60-column and 12-row tile, one to several z chunks, a single row or plane
SIZES = [(12, 10, 9), (300, 1, 2), (59, 11, 7), (60, 12, 33), (61, 13, 5), (131, 67, 45), (64, 25, 130)]


def _coef(dims, ch_varies, seed=1):
    rng = np.random.default_rng(seed)
    shape = (dims[2] + 1, dims[1] + 1, dims[0] + 1)
    ce = [(DT * rng.uniform(0.4, 1.0, shape)).astype(np.float32) for _ in range(3)]
    ch = [(DT * rng.uniform(0.4, 1.0, shape)).astype(np.float32) for _ in range(3)] if ch_varies else None
    return ce, ch


def _run(dims, ce, ch, f, calls, storage=0, stream=None, sources=None, **tuning):
    from paper_2504_09118_gb300 import Cavity
    with Cavity(*dims, DT, 1.0, ce, ch, storage, stream) as cav:
        cav.tune(**tuning)
        cav.set_fields(f)
        if sources:
            cav.set_sources(*sources)
        for n in calls:
            cav.step(n)
        assert cav.steps_done == sum(calls)
        return cav.get_fields(), cav.energy(), cav.divergence()


@pytest.mark.parametrize("dims", SIZES)
@pytest.mark.parametrize("ch_varies", [False, True])
@pytest.mark.parametrize("kernel,calls", [(0, (2,)), (0, (7,)), (3, (1, 4, 3))])
def test_f32_bitwise_equal_to_the_unfused_kernel(dims, ch_varies, kernel, calls):
    ce, ch = _coef(dims, ch_varies)
    f = ci.random_fields(21, *dims)
    got = _run(dims, ce, ch, f, calls, kernel=kernel)
    ref = _run(dims, ce, ch, f, calls, kernel=1)
    for name, a, b in zip(ci.COMPONENTS, got[0], ref[0]):
        np.testing.assert_array_equal(a, b, err_msg=name)
    assert got[1:] == ref[1:]


@pytest.mark.parametrize("stages,zchunk,graph", [(3, 0, 0), (0, 5, 1), (4, 16, 0), (0, 0, 1)])
def test_launch_shapes_bitwise(stages, zchunk, graph):
    import torch
    dims = (97, 41, 36)
    ce, ch = _coef(dims, True, 2)
    f = ci.random_fields(22, *dims)
    got = _run(dims, ce, ch, f, (37,), stream=torch.cuda.Stream(), kernel=3, stages=stages, zchunk=zchunk, use_graph=graph)
    ref = _run(dims, ce, ch, f, (37,), kernel=1)
    for a, b in zip(got[0], ref[0]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("storage,u", [(1, 2.0 ** -11), (2, 2.0 ** -8)])
@pytest.mark.parametrize("ch_varies", [False, True])
def test_16bit_error_is_that_of_one_rounding_per_two_steps(storage, u, ch_varies):
    dims, n = (75, 33, 29), 20
    ce, ch = _coef(dims, ch_varies, 3)
    f = ci.random_fields(23, *dims)
    f = [a * np.float32(s) for a, s in zip(f, (1, 1, 1, 0.01, 0.01, 0.01))]   # s_E and s_H differ
    got = _run(dims, ce, ch, f, (n,), storage=storage)[0]
    ref = _run(dims, ce, ch, f, (n,))[0]
    norm = math.sqrt(sum(float(np.sum(np.square(r, dtype=np.float64))) for r in ref))
    err = math.sqrt(sum(float(np.sum(np.square(a.astype(np.float64) - r))) for a, r in zip(got, ref)))
    assert 0 < err / norm <= 3 * u / math.sqrt(3) * math.sqrt(n / 2 + 1)


def test_currents_take_single_steps_bitwise():
    dims = (61, 25, 17)
    ce, ch = _coef(dims, True, 4)
    f = ci.random_fields(24, *dims)
    src = ([(2, 30, 12, 8), (0, 5, 5, 5)], np.random.default_rng(1).standard_normal((2, 9)).astype(np.float32))
    got = _run(dims, ce, ch, f, (6, 5), sources=src)
    ref = _run(dims, ce, ch, f, (6, 5), sources=src, kernel=1)
    for a, b in zip(got[0], ref[0]):
        np.testing.assert_array_equal(a, b)

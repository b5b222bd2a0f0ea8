"""Small cavities stepped on chip (AUTO, at least four steps a call) against the tiled kernels.

FP32 results are those of the one-step kernel bit for bit: the same operations on the same values, whatever the
split into boxes.  16-bit storage rounds once per launch instead of once per launch of one or two steps, so its
error against FP32 is bounded by the two roundings of the load and the final store, propagated by a map that
conserves the energy norm: 3 (u / sqrt 3) sqrt 2 as elsewhere.
"""
import math

import numpy as np
import pytest

import cavity_inputs as ci
from tests.gpu_util import DT

pytestmark = pytest.mark.gpu

# one cell, fewer cells than a warp, the 32-column, 16-row and 4 / 8 / 14-plane box limits and one past them,
# several boxes per axis, and the largest boxes (128 x 96 x 80 needs 32 x 16 x 14)
SIZES = [(1, 1, 1), (2, 3, 4), (32, 16, 14), (33, 17, 15), (24, 20, 17), (31, 64, 5), (64, 33, 29), (131, 67, 45),
         (7, 150, 130), (300, 40, 9), (128, 96, 80)]


def _coef(kind, dims, seed=0):
    if kind == "none":
        return None, None
    if kind == "spheres":
        return ci.sphere_coefficients(ci.sphere_list(seed + 3, 5, dims, 1.0, max(2.0, min(dims) / 3)), *dims, DT)
    # ch differs between materials too: two ce along x times three ch along z, six materials
    nx, ny, nz = dims
    rng = np.random.default_rng(seed)
    ex = rng.choice(np.array([1.0, 0.5]), size=nx + 1)[None, None, :]
    hz = rng.choice(np.array([1.0, 0.5, 0.8]), size=nz + 1)[:, None, None]
    full = [np.ascontiguousarray(np.broadcast_to(DT * v, (nz + 1, ny + 1, nx + 1)).astype(np.float32)) for v in (ex, hz)]
    return [full[0]] * 3, [full[1]] * 3


def _run(dims, coef, fields, calls, storage=0, **tuning):
    from paper_2504_09118_gb300 import Cavity
    ce, ch = coef
    with Cavity(*dims, DT, 1.0, ce, ch, storage) as cav:
        cav.tune(**tuning)
        cav.set_fields(fields)
        for n in calls:
            cav.step(n)
        assert cav.steps_done == sum(calls)
        return cav.get_fields(), cav.energy()


@pytest.mark.parametrize("dims", SIZES)
@pytest.mark.parametrize("coef", ["none", "spheres", "ch"])
@pytest.mark.parametrize("calls", [(4,), (9,), (5, 1, 6, 2)])
def test_f32_bitwise_equal_to_the_one_step_kernel(dims, coef, calls):
    c = _coef(coef, dims)
    f = ci.random_fields(11, *dims)
    got, w = _run(dims, c, f, calls)
    ref, wr = _run(dims, c, f, calls, kernel=2)
    for name, a, b in zip(ci.COMPONENTS, got, ref):
        np.testing.assert_array_equal(a, b, err_msg=name)
    assert w == wr


def test_long_calls_are_cut_into_launches_bitwise():
    dims = (40, 33, 21)
    c = _coef("spheres", dims)
    f = ci.random_fields(12, *dims)
    got, _ = _run(dims, c, f, (259, 600))
    ref, _ = _run(dims, c, f, (859,), kernel=2)
    for a, b in zip(got, ref):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("storage,u", [(1, 2.0 ** -11), (2, 2.0 ** -8)])
@pytest.mark.parametrize("dims", [(2, 3, 4), (33, 17, 15), (131, 67, 45)])
def test_16bit_rounds_at_load_and_store_only(storage, u, dims):
    c = _coef("ch", dims)
    f = ci.random_fields(13, *dims)
    got, _ = _run(dims, c, f, (64,), storage=storage)
    ref, _ = _run(dims, c, f, (64,))
    norm = math.sqrt(sum(float(np.sum(np.square(r, dtype=np.float64))) for r in ref))
    err = math.sqrt(sum(float(np.sum(np.square(a.astype(np.float64) - r))) for a, r in zip(got, ref)))
    assert 0 < err / norm <= 3 * u / math.sqrt(3) * math.sqrt(2)


@pytest.mark.parametrize("coef", ["none", "spheres"])
@pytest.mark.parametrize("dims", [(33, 17, 15), (64, 33, 29)])
def test_currents_and_probes_equal_the_per_step_launches(coef, dims):
    """Currents (two at one position, one past the end of its wave) and probes of every component, across box
    borders and several calls: fields and traces equal those of the one-step kernel with a launch per step."""
    from paper_2504_09118_gb300 import Cavity
    rng = np.random.default_rng(5)
    nx, ny, nz = dims
    src = [(0, nx // 2, ny // 2, nz // 2), (0, nx // 2, ny // 2, nz // 2), (1, nx - 1, ny - 1, nz - 1), (2, 1, 1, 0),
           (2, 32 % nx, 16 % ny, nz - 1)]
    wave = rng.standard_normal((len(src), 20)).astype(np.float32)
    probes = [(c, int(rng.integers(0, nx)), int(rng.integers(0, ny)), int(rng.integers(0, nz)))
              for c in (0, 1, 2, 3, 4, 5) for _ in range(4)] + [(0, nx // 2, ny // 2, nz // 2)]
    ce, ch = _coef(coef, dims)
    f = ci.random_fields(14, *dims)
    res = []
    for tuning in ({}, {"kernel": 2}):
        with Cavity(*dims, DT, 1.0, ce, ch) as cav:
            cav.tune(**tuning)
            cav.set_sources(src, wave)
            cav.set_fields(f)
            cav.step(3)
            cav.set_probes(probes, 22)
            for n in (5, 2, 12, 7):   # the wave and the probe buffer both end inside
                cav.step(n)
            res.append((cav.get_fields(), cav.get_probes()))
    np.testing.assert_array_equal(res[0][1], res[1][1])
    for a, b in zip(res[0][0], res[1][0]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("dims", [(32, 16, 3), (40, 33, 21), (128, 96, 80), (16, 16, 2)])
def test_a_wait_that_runs_out_ends_the_launch_and_the_context_recovers(dims):
    """One CTA waits for words that never come: the launch ends with a latched timeout, also for the CTAs that wait for
    that one; after a reload the step tags and surface buffers serve the next launches bit for bit.  (One box alone waits
    for nothing: its timeout is that of a tiled launch.)"""
    from paper_2504_09118_gb300 import Cavity, FdtdError, binding
    ce, ch = _coef("spheres", dims)
    f = ci.random_fields(15, *dims)
    want, _ = _run(dims, (ce, ch), f, (9, 600))
    with Cavity(*dims, DT, 1.0, ce, ch) as cav:
        for before in (0, 7):
            cav.set_fields(f)
            cav.step(before)
            binding.fdtd_debug_inject_timeout(cav.handle, 2000)
            cav.step(300)     # two launches on chip: the second starts with the status latched
            with pytest.raises(FdtdError) as e:
                cav.sync()
            assert e.value.code == binding.FDTD_ERR_TIMEOUT
            cav.sync()        # reported once
            cav.set_fields(f)
            cav.step(9)
            cav.step(600)
            for a, b in zip(cav.get_fields(), want):
                np.testing.assert_array_equal(a, b)

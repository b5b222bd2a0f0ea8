"""Energy and divergences against FP64 sums of the same stored state, where their two-cells-per-lane rows can go wrong:
odd and even row lengths around a lane pair and the 64-cell step, one-cell axes, one ch everywhere (the scaled sums), ch
that varies or only differs on a far face or between components (the per-cell reciprocals), per-position arrays (padding
past an odd row holds no coefficient), 16-bit storage."""
import numpy as np
import pytest

import cavity_inputs as ci
import oracle
from tests.gpu_util import DT

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (1, 3, 2), (2, 2, 2), (3, 5, 4), (63, 4, 3), (64, 3, 5), (65, 6, 3), (66, 2, 7), (129, 9, 8)]


def _coef(kind, dims):
    nx, ny, nz = dims
    shape = (nz + 1, ny + 1, nx + 1)
    rng = np.random.default_rng(sum(dims))
    flat = [np.full(shape, DT, np.float32) for _ in range(3)]
    if kind == "vacuum":
        return None, None
    ce = [np.broadcast_to(DT * rng.choice([0.5, 1.0], size=(nz + 1, 1, 1)), shape).astype(np.float32).copy() for _ in range(3)]
    if kind == "ce":
        return ce, None
    if kind == "ch flat":
        return ce, flat
    if kind == "ch face":          # the same in every cell, another value on the far x face
        flat[0][:, :, nx] *= np.float32(0.5)
        return ce, flat
    if kind == "ch components":
        flat[1] *= np.float32(0.5)
        return ce, flat
    if kind == "ch varies":
        return ce, [np.broadcast_to(DT * rng.choice([0.5, 1.0], size=(1, ny + 1, 1)), shape).astype(np.float32).copy()
                    for _ in range(3)]
    full = [(DT * rng.uniform(0.4, 1.0, shape)).astype(np.float32) for _ in range(6)]
    return full[:3], (full[3:] if kind == "full" else None)


@pytest.mark.parametrize("dims", SIZES)
@pytest.mark.parametrize("kind", ["vacuum", "ce", "ch flat", "ch face", "ch components", "ch varies", "full", "full ce"])
@pytest.mark.parametrize("storage", [0, 1])
def test_equal_the_fp64_sums_of_the_stored_state(dims, kind, storage):
    from paper_2504_09118_gb300 import Cavity
    ce, ch = _coef(kind, dims)
    with Cavity(*dims, DT, 1.0, ce, ch, storage) as cav:
        cav.set_fields(ci.random_fields(41, *dims))
        got = np.array([cav.energy(), *cav.divergence()])
        stored = oracle.as_f64(cav.get_fields())     # what the sums are taken of
    vac = float(np.float32(DT))
    c64 = [vac if c is None else [a.astype(np.float64) for a in c] for c in (ce, ch)]
    de, dh = oracle.divergence(stored, *c64)
    ref = np.array([oracle.energy(stored, *c64, DT), np.linalg.norm(de), np.linalg.norm(dh)])
    # terms to about 2^-48 each, summed without cancellation beyond the state's own size
    scale = np.maximum(np.abs(ref), 1e-3 * np.abs(ref).max())
    assert np.all(np.abs(got - ref) <= 1e-12 * scale), (got, ref)


@pytest.mark.parametrize("storage,scale", [(0, 1.0), (0, 2.0 ** -36), (1, 1.0)])
@pytest.mark.parametrize("dims", [(33, 12, 9), (64, 5, 4)])
def test_divergence_of_a_divergence_free_field(dims, storage, scale):
    """H = curl E of a few steps from H = 0, in SI units (ch about 1e-3), also of a weak field: the six values of a cell
    cancel but for their own roundings, which is what the divergence measures.  A cell's sum is exact to a few 2^-48 of
    its terms, and so is the norm over the cells."""
    from paper_2504_09118_gb300 import Cavity
    dx, dt = 1e-3, 1.9e-12
    full = [np.full(tuple(n + 1 for n in reversed(dims)), v, np.float32)
            for v in (dt / (8.8541878128e-12 * dx), dt / (1.25663706212e-6 * dx))]
    f = [a * np.float32(scale if c < 3 else 0.0) for c, a in enumerate(ci.random_fields(43, *dims))]
    with Cavity(*dims, dt, dx, full[:1] * 3, full[1:] * 3, storage) as cav:
        cav.set_fields(f)
        cav.step(3)
        got = cav.divergence()[1]
        stored = oracle.as_f64(cav.get_fields())
    c64 = [[v.astype(np.float64)] * 3 for v in full]
    ref = np.linalg.norm(oracle.divergence(stored, *c64)[1])
    terms = sum(float(np.linalg.norm(a)) for a in stored[3:]) / float(full[1].flat[0])
    assert ref > 0 and abs(got - ref) <= 8 * 2.0 ** -48 * terms, (got, ref)

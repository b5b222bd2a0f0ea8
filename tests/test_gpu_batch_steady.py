"""Batches of members with every coefficient layout in one launch (uniform, PEC-coded ids with uniform and varying ch,
more than 31 materials): the default launch shape and tile heights with and without steady-state plane bodies, z-lengths
down to tiles without a steady plane, own (odd) step counts that end in one-step stores.  FP32 members equal the same
cavity stepped alone by the one-step kernel bit for bit."""
import numpy as np
import pytest

import cavity_inputs as ci
from tests.gpu_util import DT

pytestmark = pytest.mark.gpu

DIMS = [(60, 12, 40), (61, 13, 5), (16, 30, 1), (90, 40, 33), (33, 25, 70), (7, 5, 3), (96, 24, 17), (20, 66, 2)]


def _coef(n, dims):
    nx, ny, nz = dims
    shape = (nz + 1, ny + 1, nx + 1)
    rng = np.random.default_rng(n)

    def layers(values, axis):
        v = rng.choice(np.array(values), size=shape[axis])
        v = v.reshape([-1 if a == axis else 1 for a in range(3)])
        return [np.ascontiguousarray(np.broadcast_to(DT * v, shape).astype(np.float32))] * 3

    kind = n % 4
    if kind == 0:
        return None, None                                    # uniform
    if kind == 1:
        return layers([1.0, 0.5], 2), None                   # ids, uniform ch
    if kind == 2:
        return layers([1.0, 0.5], 1), layers([1.0, 0.7], 2)  # ids, ch varies
    # up to 49 materials (more than 31 where the sides allow): ids without PEC coding
    return layers(np.linspace(0.4, 1.0, 7), 2), layers(np.linspace(0.5, 1.0, 7), 1)


@pytest.fixture(scope="module")
def members():
    return [(d, *_coef(n, d), ci.random_fields(200 + n, *d)) for n, d in enumerate(DIMS)]


@pytest.fixture(scope="module")
def alone(members):
    """Fields of each member after every step count used below, stepped alone by the one-step kernel."""
    from paper_2504_09118_gb300 import Cavity
    out = []
    for d, ce, ch, f in members:
        with Cavity(*d, DT, 1.0, ce, ch) as cav:
            cav.tune(kernel=2)
            cav.set_fields(f)
            got = {}
            for n in range(1, 22):
                cav.step(1)
                got[n] = cav.get_fields()
        out.append(got)
    return out


@pytest.mark.parametrize("tuning", [{}, dict(kernel=3, tile_y=12, zchunk=1), dict(kernel=3, tile_y=12, zchunk=4),
                                    dict(kernel=3, tile_y=8, zchunk=9), dict(kernel=3, tile_y=16), dict(kernel=4)])
@pytest.mark.parametrize("own", [False, True])
@pytest.mark.parametrize("graph", [0, 1])
def test_members_equal_alone_bitwise(members, alone, tuning, own, graph):
    import torch
    from paper_2504_09118_gb300 import Cavity
    from paper_2504_09118_gb300 import binding as B
    s = torch.cuda.Stream()
    b = B.fdtd_batch_create(0, s)
    cavs = []
    try:
        B.fdtd_batch_set_tuning(b, use_graph=graph, **tuning)
        for n, (d, ce, ch, f) in enumerate(members):
            cav = Cavity(*d, DT, 1.0, ce, ch, 0, s)
            cav.set_fields(f)
            B.fdtd_batch_add(b, cav.handle)
            if own:
                B.fdtd_batch_set_steps(b, cav.handle, 21 - 2 * n - (n % 2))
            cavs.append(cav)
        B.fdtd_batch_step(b, 18)
        B.fdtd_batch_step(b, 3)
        B.fdtd_batch_sync(b)
        for n, cav in enumerate(cavs):
            B.fdtd_batch_remove(b, cav.handle)
            steps = 21 - 2 * n - (n % 2) if own else 21
            assert cav.steps_done == steps
            for name, x, y in zip(ci.COMPONENTS, cav.get_fields(), alone[n][steps]):
                np.testing.assert_array_equal(x, y, err_msg=f"{DIMS[n]} {name}")
    finally:
        B.fdtd_batch_destroy(b)
        for cav in cavs:
            cav.close()

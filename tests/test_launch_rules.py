"""Rules that choose between launches, on the CPU through the library's host-only entry points."""
import itertools
import random

import pytest

from paper_2504_09118_gb300 import binding as B


def test_exchange_kernel_only_on_the_current_device():
    """A kernel launch goes to the current device, and on the default stream to that device's: slabs that live elsewhere
    take the copies, ordered by events even when both name the same stream handle."""
    for lo, hi, cur, same in itertools.product(range(3), range(3), range(3), (False, True)):
        kernel, events = B.fdtd_debug_exchange_route(lo, hi, cur, same)
        assert kernel == (lo == hi == cur)
        assert events == (not kernel or not same)


SMS = 152
DEPTHS = (2, 4, 6, 8, 11, 14)   # planes of the on-chip kernel's instances


def depth(nz, pz):
    return next((d for d in DEPTHS if d >= -(-nz // pz)), None)


def splits(dims, most):
    """Every split into boxes of at most 32 x 16 x 14 cells, as (instance depth, boxes)."""
    nx, ny, nz = dims
    for px in range(-(-nx // 32), min(nx, most) + 1):
        for py in range(-(-ny // 16), min(ny, most // px) + 1):
            for pz in range(1, min(nz, most // (px * py)) + 1):
                if depth(nz, pz):
                    yield depth(nz, pz), px * py * pz


def sizes():
    rng = random.Random(4)
    fixed = [(1, 1, 1), (16, 16, 16), (24, 20, 17), (32, 32, 32), (131, 67, 45), (128, 96, 80), (7, 150, 130), (300, 40, 9),
             (129, 97, 90), (1, 2433, 1), (1, 2432, 14)]
    return fixed + [tuple(int(10 ** rng.uniform(0, 2.2)) for _ in range(3)) for _ in range(24)]


@pytest.mark.parametrize("dims", sizes())
def test_resident_split_takes_the_least_depth_then_the_fewest_boxes(dims):
    parts = B.fdtd_debug_resident_split(*dims, SMS)
    every = list(splits(dims, SMS))
    if not every:
        assert parts is None
        return
    px, py, pz = parts
    assert -(-dims[0] // px) <= 32 and -(-dims[1] // py) <= 16
    assert (depth(dims[2], pz), px * py * pz) == min(every)


def test_small_cavities_leave_room_for_other_launches():
    """Eight contexts of up to 24 x 20 x 17 cells, or four of 32^3, fit on the SMs at once."""
    for dims, most in (((16, 16, 16), SMS // 8), ((24, 20, 17), SMS // 8), ((32, 32, 32), SMS // 4)):
        px, py, pz = B.fdtd_debug_resident_split(*dims, SMS)
        assert px * py * pz <= most


# cavities where a height is ahead of both others by 4 % or more (us per step with 8, 12 and 16 rows, FP32)
HEIGHTS = [((474, 184, 230), 16), ((160, 150, 140), 16), ((482, 195, 147), 16), ((305, 311, 274), 16), ((230, 850, 340), 16),
           ((172, 143, 50), 12), ((243, 69, 75), 12), ((164, 499, 124), 12), ((459, 227, 270), 12), ((55, 31, 32), 8)]


@pytest.mark.parametrize("dims,rows", HEIGHTS)
def test_two_step_height_is_the_measured_best(dims, rows):
    assert B.fdtd_debug_two_step_shape(*dims, B.FDTD_F32, SMS)[0] == rows


def test_two_step_ring_depth_by_size():
    """Both sides of the sizes from which FP32 rings are shallower; 16-bit rings always fill the shared memory."""
    shape = lambda dims, storage=B.FDTD_F32: B.fdtd_debug_two_step_shape(*dims, storage, SMS)
    assert shape((512, 512, 512)) == (12, 5)
    assert shape((323, 263, 844)) == (12, 5)          # 7.2e7 cells
    assert shape((459, 227, 270)) == (12, 0)          # 2.8e7
    assert shape((512, 512, 256)) == (16, 0)          # 6.7e7
    for dims in ((512, 512, 512), (323, 263, 844), (459, 227, 270)):
        for storage in (B.FDTD_F16, B.FDTD_BF16):
            assert shape(dims, storage)[1] == 0
    for storage in (B.FDTD_F32, B.FDTD_BF16):         # one cell to the largest axes
        for dims in ((1, 1, 1), (1, 1, 32768), (32768, 1, 1), (1, 32768, 3), (61, 17, 5)):
            assert shape(dims, storage)[0] in (8, 12, 16)

"""Layout conversion and the storage-scale scan at the edges of their blocks and planes.

Loading and reading back without a step is exact: FP32 values come back bit for bit inside each extent, 16-bit
ones as the storage rounding of the scaled value, and entries outside an extent as 0, whatever they held.  The
scale is set by the largest magnitude of each field's extent, wherever it sits.
"""
import numpy as np
import pytest

import cavity_inputs as ci

pytestmark = pytest.mark.gpu

# one cell, one column, rows and planes around the 256-entry block, the 4-plane group and the 128-entry row scan
SIZES = [(1, 1, 1), (1, 7, 3), (5, 1, 4), (31, 8, 2), (32, 7, 3), (96, 2, 5), (127, 3, 1), (129, 5, 6), (255, 1, 7)]


def _state(dims, seed=0):
    """Fields with garbage outside each extent, and the same with what a load keeps."""
    nx, ny, nz = dims
    full = [ci.uniform_pm1(seed, c, (nx + 1) * (ny + 1) * (nz + 1)).reshape(nz + 1, ny + 1, nx + 1) for c in range(6)]
    kept = []
    for c, name in enumerate(ci.COMPONENTS):
        f = full[c].copy()
        f[~ci.extent_mask(name, *dims)] = 0.0
        if name[0] == "E":
            f[ci.tangential_e_mask(name, *dims)] = 0.0
        kept.append(f)
    return full, kept


# host arrays just below and above the sizes up to which the kernels write (1 MiB) and read (16 MiB) them directly
DIRECT = [(34, 34, 33), (35, 35, 35), (88, 88, 87), (88, 88, 88)]


@pytest.mark.parametrize("dims", SIZES + DIRECT)
@pytest.mark.parametrize("device", [False, True])
def test_load_and_read_back_f32_exact(dims, device):
    import torch
    from paper_2504_09118_gb300 import Cavity
    full, kept = _state(dims)
    with Cavity(*dims, ci.COURANT_HALF_DT) as cav:
        if device:
            cav.set_fields([torch.from_numpy(f).cuda() for f in full], on_device=True)
            out = [torch.full(cav.shape, 7.0, device="cuda") for _ in range(6)]
            got = [t.cpu().numpy() for t in cav.get_fields(out, on_device=True)]
        else:
            cav.set_fields(full)
            got = cav.get_fields()
    for c in range(6):
        np.testing.assert_array_equal(got[c], kept[c])


@pytest.mark.parametrize("dims", SIZES)
@pytest.mark.parametrize("where", ["first", "last"])
def test_f16_scale_follows_the_largest_entry_of_the_extents(dims, where):
    """The scale is 2^(8 - ceil(log2 max)) with max over the extents: a large value at the first or last entry of
    one component's extent moves it, garbage outside the extents does not."""
    import torch
    from paper_2504_09118_gb300 import Cavity
    from paper_2504_09118_gb300 import binding as B
    full, _ = _state(dims, 3)
    for comp in (2, 4):   # Ez (rows to nx, planes to nz - 1), Hy (rows to nx - 1, planes to nz - 1)
        name = ci.COMPONENTS[comp]
        f = [a * np.float32(0.25) for a in full]
        m = ci.extent_mask(name, *dims)
        idx = tuple(v[0 if where == "first" else -1] for v in np.nonzero(m))
        f[comp][idx] = 37.0
        for c in range(6):   # outside the extents: ignored
            f[c][~ci.extent_mask(ci.COMPONENTS[c], *dims)] = 5000.0
        mx = [max(float(np.abs(f[c][ci.extent_mask(ci.COMPONENTS[c], *dims)]).max()) for c in g)
              for g in ((0, 1, 2), (3, 4, 5))]
        s = [B.fdtd_storage_scale_of(v) for v in mx]
        with Cavity(*dims, ci.COURANT_HALF_DT, storage=B.FDTD_F16) as cav:
            cav.set_fields([torch.from_numpy(a).cuda() for a in f], on_device=True)
            dev = cav.get_fields()
            cav.set_fields(f)
            host = cav.get_fields()
        for c in range(6):
            cm = ci.extent_mask(ci.COMPONENTS[c], *dims)
            ref = f[c].copy()
            ref[~cm] = 0.0
            if c < 3:
                ref[ci.tangential_e_mask(ci.COMPONENTS[c], *dims)] = 0.0
            sc = np.float32(s[c // 3])
            ref = (ref * sc).astype(np.float16).astype(np.float32) / sc
            np.testing.assert_array_equal(dev[c], ref)
            np.testing.assert_array_equal(host[c], ref)


@pytest.mark.parametrize("tuning", [{}, dict(kernel=2, use_graph=1), dict(kernel=3, use_graph=1)])
@pytest.mark.parametrize("storage", [1, 2])
def test_reloads_with_equal_and_other_scales_match_a_fresh_context(tuning, storage):
    """The folded coefficients and launch records of a 16-bit context are rebuilt only when s_E / s_H changes: each of a
    series of loads (another ratio, back, the same, both scales times 4 with a current set) steps as in a new context."""
    import torch
    from paper_2504_09118_gb300 import Cavity
    dims = (61, 30, 21)
    ce, ch = ci.sphere_coefficients(ci.sphere_list(9, 4, dims, 3.0, 9.0), *dims, ci.COURANT_HALF_DT)
    base = ci.random_fields(31, *dims)
    src = [(2, 30, 15, 10)], np.linspace(0.1, 1.0, 40, dtype=np.float32)[None]
    s = torch.cuda.Stream()

    def solve(cav, e, h, sources):
        cav.set_sources(*(src if sources else ([], [])))
        cav.set_fields([a * np.float32(e if c < 3 else h) for c, a in enumerate(base)])
        cav.step(19)
        return cav.get_fields()

    with Cavity(*dims, ci.COURANT_HALF_DT, 1.0, ce, ch, storage, s) as cav:
        cav.tune(**tuning)
        for e, h, sources in ((1, 1, 0), (8, 1, 0), (1, 1, 0), (1, 1, 0), (1, 1, 1), (4, 4, 1), (1, 0.5, 1)):
            got = solve(cav, e, h, sources)
            with Cavity(*dims, ci.COURANT_HALF_DT, 1.0, ce, ch, storage, s) as fresh:
                fresh.tune(**tuning)
                want = solve(fresh, e, h, sources)
            for a, b in zip(got, want):
                np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("offset", [1, 2, 3])
@pytest.mark.parametrize("storage", [0, 1, 2])
def test_host_arrays_at_any_address(offset, storage):
    """Views into packed buffers, contiguous but not at a multiple of 4 bytes: one such array among six, and all six, load
    and read back like aligned ones."""
    from paper_2504_09118_gb300 import Cavity
    dims = (9, 8, 7)
    shape = tuple(n + 1 for n in reversed(dims))
    full, _ = _state(dims, 5)

    def view(a=None):
        raw = np.zeros(4 * int(np.prod(shape)) + 8, np.uint8)
        v = np.frombuffer(raw.data, np.float32, int(np.prod(shape)), offset + (-raw.ctypes.data) % 4).reshape(shape)
        assert v.ctypes.data % 4 == offset and v.flags.c_contiguous and v.flags.writeable
        if a is not None:
            v[:] = a
        return v

    with Cavity(*dims, ci.COURANT_HALF_DT, storage=storage) as cav:
        cav.set_fields(full)
        want = cav.get_fields()
        for which in (range(6), [4]):
            cav.set_fields([view(a) if c in which else a for c, a in enumerate(full)])
            out = [view() if c in which else np.empty(shape, np.float32) for c in range(6)]
            cav.get_fields(out)
            for a, b in zip(out, want):
                np.testing.assert_array_equal(a, b)

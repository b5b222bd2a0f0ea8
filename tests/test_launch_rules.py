"""Rules that choose between launches, on the CPU through the library's host-only entry points."""
import itertools

from paper_2504_09118_gb300 import binding as B


def test_exchange_kernel_only_on_the_current_device():
    """A kernel launch goes to the current device, and on the default stream to that device's: slabs that live elsewhere
    take the copies, ordered by events even when both name the same stream handle."""
    for lo, hi, cur, same in itertools.product(range(3), range(3), range(3), (False, True)):
        kernel, events = B.fdtd_debug_exchange_route(lo, hi, cur, same)
        assert kernel == (lo == hi == cur)
        assert events == (not kernel or not same)

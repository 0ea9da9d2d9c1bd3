"""The bounded waits of the U-Net's tcgen05 kernels (needs a GB300): a warp whose lanes poll a
barrier leaves the wait as a whole when the polls of one lane run out, and goes on as a whole
otherwise.  The barrier of this check always completes, so every lane's loop ends."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("polls", [1000, 1 << 20])
def test_a_warp_gives_up_as_one(polls):
    from paper_2306_11320_gb300.unet import net_library

    lib = net_library()
    out = (C.c_int * 4)(-1, -1, -1, -1)
    assert lib.tpfnet_check_bounded_wait(polls, out) == 0
    assert list(out) == [0, 0, 32, 1]
    assert lib.tpfnet_check_bounded_wait(0, out) != 0
    assert lib.tpfnet_status() == 0  # the check raises a flag of its own

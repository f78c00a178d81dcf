"""How many passes over the network a first call takes to choose its kernels, on a
runtime without a device."""
import pytest
from host_runtime import run


@pytest.mark.parametrize("widths,lin,passes", [
    ([2, 20, 20, 1], 0, 1),          # nothing to choose: one pass finds that out
    ([8, 20, 20, 1], 0, 1),
    ([1, 20, 20, 1], 0, 1),
    ([3, 64, 64, 64, 1], 0, 10),     # the wide affine steps
    ([6, 64, 64, 1], 0, 10),
    ([3, 32, 32, 32, 32, 1], 4, 10)])   # and enclosures on grids (order 16)
def test_passes_of_a_first_call(tmp_path, widths, lin, passes):
    run(tmp_path, """
widths, lin, passes, B = %r, %r, %r, 40
host = [np.zeros((widths[i + 1], widths[i] + 1), np.float32) for i in range(len(widths) - 1)]
net, keep = bern.make_net(widths, [x.ctypes.data for x in host], [x.ctypes.data for x in host])
plan, keep2 = bern.make_plan(2, widths, 16, 0.0, 0, lin)
boxes = np.zeros((B, widths[0], 2), np.float32)
res = bern.bern_result(empty(4 * B), empty(4 * B), empty(8 * B), None, None, 0)
h = context()
def launches(on):
    k = lib.bern_kernel_launches(h)
    assert lib.bern_set_autotune(h, on) == 0
    assert lib.bern_propagate(h, ctypes.byref(net), boxes.ctypes.data, B, ctypes.byref(plan),
                              ctypes.byref(res)) == 0
    return lib.bern_kernel_launches(h) - k
one = launches(0)
# a pass may hold a kernel more where a variant leaves the stability screen to its own
first, again = launches(1), launches(1)
assert again <= one + (len(widths) if passes > 1 else 0), (again, one)
assert first <= (passes + 1) * (one + (len(widths) if passes > 1 else 0)), (first, one)
""" % (widths, lin, passes))

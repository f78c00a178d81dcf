"""Which kernels a call takes where the choice follows from its sizes alone, on a
runtime without a device (152 multiprocessors)."""
import pytest
from host_runtime import run


@pytest.mark.parametrize("h_in,h_out,rows,boxes,kernel", [
    (128, 200, 165, 1, "8k_affineI"), (128, 200, 165, 300, "8k_affineI"),
    (128, 200, 165, 3000, "k_affine_wide"), (128, 200, 17, 30, "8k_affineI"),
    (64, 64, 165, 1, "k_affine_wide"), (100, 200, 33, 1, "k_affine_wide"),
    (300, 200, 33, 3000, "8k_affineI")])
def test_affine(tmp_path, h_in, h_out, rows, boxes, kernel):
    """Weights that nearly fill shared memory leave a box to one block: only
    batches take the register-blocked kernel then, single boxes are tiled."""
    run(tmp_path, """
h = context()
launched()
assert lib.bern_affine(h, %d, %d, %d, empty(8), empty(8), empty(8), empty(8), %d, empty(8),
                       empty(8), empty(8), %d, empty(8)) == 0
names = launched()
assert len(names) == 1 and %r in names[0], names
""" % (boxes, h_out, h_in, rows, rows, kernel))

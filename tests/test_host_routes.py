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


@pytest.mark.parametrize("n,l,kernels", [
    (4, 10, "enclose"), (5, 10, "k_enclose_big"), (4, 9, "k_enclose_slab"), (5, 9, "k_enclose_slab"),
    (6, 9, "k_enclose_slab"), (7, 4, "k_enclose_expand"), (8, 3, "k_enclose_expand"),
    (8, 4, "k_enclose_slab"), (6, 5, "k_enclose_slab"), (4, 8, "k_enclose_expand")])
def test_enclose(tmp_path, n, l, kernels):
    """Orders and variables at the ends of the enclosure's forms."""
    run(tmp_path, """
h = context()
n, l = %d, %d
assert lib.bern_enclose(h, n, 2, 3, l, 0, empty(8), empty(8), bern.num_monomials(n, l), empty(8),
                        empty(8), empty(8)) == 0
names = launched()
assert len(names) == 1 and %r in names[0], names
assert l < 10 or "slab" not in names[0], names
""" % (n, l, kernels))

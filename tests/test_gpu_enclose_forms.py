"""Enclosures in seven and eight variables whose levels take more than a quarter of a
multiprocessor's shared memory: a block per item."""
import pytest

from test_gpu_enclose_orders import test_enclose_orders as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,l,D,B,h", [(7, 4, 4, 2, 3), (7, 4, 5, 1, 2), (8, 3, 3, 2, 3),
                                       (8, 3, 4, 1, 2), (5, 7, 7, 1, 3)])
def test_one_item_to_a_block(n, l, D, B, h):
    check(n, l, D, B, h)

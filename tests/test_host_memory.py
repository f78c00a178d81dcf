"""What a call does when device memory is short, on a runtime without a device."""
from host_runtime import run

COMPOSE = """
def compose(h, n, D, B, hh, d=2, degrees=False):
    M = bern.num_monomials(n, D)
    keep = bern.num_monomials(n, min(2 * D, 16))
    items = B * hh
    launched()
    rc = lib.bern_compose(h, n, B, hh, 16, 0.0, empty(items), empty(items * 4 * bern.COEF_STRIDE),
                          empty(items * 4), empty(items) if degrees else None, d,
                          empty(items * 4), empty(items * 4), empty(8), empty(8), M,
                          empty(items * 4), empty(8), empty(8), keep, empty(items * 4))
    sizes.append(allocated())
    return rc, launched()
sizes = []                                            # of each call
def count(names, what):
    return sum(what in x for x in names)
"""


def test_squares_without_their_scratch_take_the_pair_lists(tmp_path):
    """Inputs past shared memory (five variables, degree 8: 1287 terms): with no
    scratch to be had the call goes on with the pair lists, with room for some of
    the groups it takes several passes, and each state serves the calls after it."""
    run(tmp_path, COMPOSE + """
h = context()
rc, k = compose(h, 5, 8, 4, 64)                       # eight groups and eight spare
assert rc == 0 and count(k, "k_square_units") == 1, (rc, k)
lib.bern_destroy(h)

h = context()
rc, k = compose(h, 5, 8, 4, 64, d=1)                  # tables and queues
assert rc == 0 and count(k, "k_square") == 0, (rc, k)
rt.host_set_alloc_limit(300 << 10)                    # less than a group of 400 KB
for _ in range(2):
    rc, k = compose(h, 5, 8, 4, 64)
    assert rc == 0 and count(k, "k_square_units") == 0 and count(k, "k_compose_pairs") == 1, (rc, k)
rt.host_set_alloc_limit(2 << 20)                      # a few groups
for _ in range(2):
    rc, k = compose(h, 5, 8, 4, 64)
    assert rc == 0 and count(k, "k_square_units") > 1, (rc, k)
rt.host_set_alloc_limit(1 << 40)
rc, k = compose(h, 5, 8, 64, 64)                      # more items: asked for again
assert rc == 0 and count(k, "k_square_units") == 1, (rc, k)
lib.bern_destroy(h)
""")


def test_no_scratch_where_nothing_is_squared(tmp_path):
    """Order 3 for every neuron has no squares; per-neuron orders up to 3 may have."""
    run(tmp_path, COMPOSE + """
def sizes_of(d, degrees):
    h = context()
    assert compose(h, 5, 7, 4, 64, d=1)[0] == 0       # 792 terms: tables and queues
    assert compose(h, 5, 7, 4, 64, d=d, degrees=degrees)[0] == 0
    lib.bern_destroy(h)
    return sizes[-1]
scratch, = sizes_of(2, False)
assert scratch in sizes_of(3, True)
assert scratch not in sizes_of(3, False)
""")


def test_tables_whose_copy_failed_are_built_again(tmp_path):
    """A copy of a table to the device fails, the first, the last or any between: the
    call says so, and the next one does not run on what is there."""
    run(tmp_path, COMPOSE + """
def tries(n, D, d):
    h = context()
    rt.host_count_copies()
    rc, k = compose(h, n, D, 1, 3, d=d)
    total = rt.host_count_copies()
    assert rc == 0 and total > 10
    lib.bern_destroy(h)
    for left in sorted({0, 1, total // 3, total // 2, total - 2, total - 1}):
        h = context()
        launched()
        rt.host_fail_copies_after(left)
        rc, k = compose(h, n, D, 1, 3, d=d)
        assert rc != 0 and not k, (left, rc, k)
        rt.host_fail_copies_after(-1)
        first = rt.host_count_copies()
        rc, k = compose(h, n, D, 1, 3, d=d)
        assert rc == 0 and k, (left, rc, k)
        # what a failed build had copied is copied again; the product tables of order
        # 3 that were complete stay
        again = rt.host_count_copies()
        assert again >= total - 1 if d == 2 else first + again >= total, (left, total, first, again)
        rc, k = compose(h, n, D, 1, 3, d=d)
        assert rc == 0 and rt.host_count_copies() == 0
        lib.bern_destroy(h)
tries(4, 2, 2)
tries(2, 2, 3)
""")

"""bench.py's operation count of a timed slice follows the walk that the slice
takes: from n = 13 on tiles where 10 + n + delta variables vary, else the
dense walk (a 2^38-term slice of L(31) had been booked at 12 instead of 92
operations a term)."""
import bench


def test_operations_of_a_slice():
    for variant, n, bits, skips in ((1, 31, 38, False), (1, 31, 41, False), (1, 31, 42, True),
                                    (0, 28, 37, False), (0, 28, 38, True), (2, 30, 40, True),
                                    (0, 12, 23, False)):
        want = bench.skip_ops_per_term(variant, n) if skips else bench.alg_ops_per_term(variant, n)
        assert bench.slice_ops_per_term(variant, n, bits) == want
    assert bench.alg_ops_per_term(1, 31) == 92 and bench.skip_ops_per_term(1, 31) < 13


def test_a_slice_is_no_larger_than_the_count():
    # S(21) with Lemma 2.4: 2^26 items of 2^14 terms (a 2^42-term slice had
    # been timed over the count's 2^40 terms and booked whole)
    assert bench.slice_items(1 << 26, 14, 42) == 1 << 26
    assert bench.slice_items(1 << 26, 14, 38) == 1 << 24
    assert bench.slice_items(1 << 20, 25, 22) == 1

"""The confidence bound sums only the terms that count and compares only near its root; it must still return the very
double of the plain bisection over all terms (the oracle's), at the ends of its ranges too."""
import pytest

import oracle
import paper_2108_09413_b200 as isc


@pytest.mark.parametrize("alpha", [1e-300, 1e-12, 0.001, 0.5, 0.999])       # a root far below k / n, near it, above it
@pytest.mark.parametrize("N,ks", [(1, (0, 1)), (2, (1,)), (3, (1, 2)), (17, (1, 8, 16)), (1000, (1, 2, 501, 998, 999)),
                                  (20000, (1, 9999, 10001, 19000, 19999))])
def test_bound_and_test_equal_the_full_sums(N, ks, alpha):
    for k in ks:
        counts = [k, (N - k) // 2, N - k - (N - k) // 2]
        assert isc.certify_decide([1, 0, 0], counts, N, 0.25, alpha) == oracle.certify_decide([1, 0, 0], counts, N, 0.25, alpha)
        assert isc.predict_decide(counts, alpha) == oracle.predict_decide(counts, alpha)
        for two_sided in (False, True):
            assert isc.certify_integer_decide([1, 0, 0], counts, N, 0.25, alpha, two_sided) == \
                oracle.certify_integer_decide([1, 0, 0], counts, N, 0.25, alpha, two_sided)

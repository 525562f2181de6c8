"""The automatic choice between the dense and the sorting quotient: the same CSR on both sides of the rule."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [12.0, 15.0, 22.0])  # R-MAT 20 (31M entries): k about 3,300, 4,200 and 6,000
def test_auto_equals_sort(tau):
    import paper_1506_03265_gb300 as cd
    e = inputs.rmat(20, 16, 1 << 20, 2)
    g = cd.build_csr(e.src, e.dst, e.w, e.n)
    auto, sort = (cd.quotient_build(cd.cluster(g, tau, 1, quotient_mode=m))
                  for m in (cd.QUOTIENT_AUTO, cd.QUOTIENT_SORT))
    assert auto.info() == sort.info() and auto.info()[0] > 2000
    for a, b in zip(auto.copy(), sort.copy()):
        assert np.array_equal(a, b)
    cd.tuning_set(dense_quotient_k=1024)  # a lowered knob keeps the sort
    try:
        low = cd.quotient_build(auto.clustering)
    finally:
        cd.tuning_set()
    for a, b in zip(low.copy(), sort.copy()):
        assert np.array_equal(a, b)

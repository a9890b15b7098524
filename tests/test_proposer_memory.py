"""Every allocation of the proposer's workspace in turn fails while it grows for
a larger graph: the call reports it, and calls on the graph before and on the
larger one give what they gave."""
import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu


def test_failed_growth_leaves_a_usable_proposer():
    import paper_1808_05458_gb300 as mc
    small, large = graphgen.random_connected(300, 1500, seed=31, wmax=9), graphgen.rhg(9, 1 << 11, 24.0)
    with mc.Graph(*small) as A, mc.Graph(*large) as B:
        P = mc.Proposer(seed=3)
        want_b = P.forward(B)
        P.close()
        for k in range(12):
            P = mc.Proposer(seed=3)
            want_a = P.forward(A)
            try:
                mc.test_fail_alloc_after(k)
                with pytest.raises(mc.MinCutError) as e:
                    P.forward(B)
            finally:
                mc.test_fail_alloc_after(-1)
            assert e.value.code == mc.MC_ENOMEM
            assert np.array_equal(P.forward(A), want_a)
            assert np.array_equal(P.forward(B), want_b)
            P.close()

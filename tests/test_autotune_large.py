"""Autotuning a batch large enough to be copied in chunks, from pageable
arrays: the choice is by the kernels' time and not by the copies', so that the
block-per-graph solver, faster than any shape of the warps on this batch
whatever the link, stays chosen."""
import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu


def test_choice_leaves_the_copies_out():
    import paper_1808_05458_gb300 as mc
    b = [np.array(x) for x in graphgen.batch(1, 4096, 50, 2000, 4, 16, 100)]
    assert len(b[1]) >= 32 << 20
    mc.batch_set_shape(-1)
    want = mc.batch_min_cut(*b)[0]
    try:
        mc.batch_autotune(*b)
        for _ in range(2):
            lam, _, _, st = mc.batch_min_cut(*b)
            assert (lam == want).all()
        # the default's chunks are several launches a call, a shape's at most one
        assert st["kernel_launches"] > 1
    finally:
        mc.batch_set_shape(-1)

"""Under a node budget or a stack limit that some rays exceed, a batch's megakernel gives the chains, counters
and status of the chain set's own: it visits the nodes in the same order.  (The wavefront's kernels trace
speculatively, past a leaf that waits to be tested, and so stop other rays.)"""
import numpy as np
import pytest

from paper_2409_07148_gb300 import jr, scenes

pytestmark = pytest.mark.gpu


def _run(scene, sc, mode, limits, flags):
    ch = jr.Chains(scene, sc.width, sc.height, sc.depth, 3000, seed=6, flags=flags, burn_in=0)
    ch.set_limits(*limits)
    if isinstance(mode, int):
        batch = jr.Batch([ch])
        batch.set_block(mode)
        batch.advance(6)
    else:
        ch.set_execution(mode)
        ch.advance(6)
    st = ch.stats(check=False)
    st.pop("p_sum_large")
    return st, *ch.get_state()


# 14 visits and 4 entries: some rays exceed each.  "mega": 3000 chains, a few per warp; batch blocks of 32 and 256
# chains
@pytest.mark.parametrize("limits,bit", [((14, 0), jr.JR_STATUS_TRAVERSAL), ((0, 4), jr.JR_STATUS_STACK)])
@pytest.mark.parametrize("flags", [0, jr.JR_FLAG_MH])
def test_limits_stop_the_same_rays_in_a_batch(limits, bit, flags):
    sc = scenes.random_boxes(5, 5000, 64, 48, 6)
    scene = jr.Scene(sc)
    ref = _run(scene, sc, "mega", limits, flags)
    assert ref[0]["status_word"] & bit
    for mode in (32, 256):
        got = _run(scene, sc, mode, limits, flags)
        assert got[0] == ref[0], mode
        assert np.array_equal(got[1], ref[1]) and np.array_equal(got[2], ref[2]), mode

"""What look-ahead holds: one buffer of at most 128 MB of F where no window's tail is put off, and an
older, smaller one where a larger cannot be had."""
import numpy as np
import pytest

from paper_2409_07148_gb300 import jr, scenes

pytestmark = pytest.mark.gpu

MB = 1 << 20


# windows of 2^23 paths: 256 steps of 2^15 chains, 2^15 of 256; a call of more steps has a second window
@pytest.mark.parametrize("name,n,steps,flags", [("spheres", 1 << 15, 300, jr.JR_FLAG_MALA), ("box", 256, 33000, 0)])
def test_no_second_buffer_where_no_tail_waits(name, n, steps, flags):
    import torch
    sc = scenes.cornell(width=16, height=16, depth=1) if name == "box" else \
        scenes.cornell_spheres(width=16, height=16, depth=2, n_lon=24, n_lat=25)
    ch = jr.Chains(jr.Scene(sc), sc.width, sc.height, sc.depth, n, seed=5, flags=flags, c_tilde=10.0)
    ch.advance(1)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    launches = ch.advance_timed(steps)["path"]["launches"]
    assert launches == 2
    held = before - torch.cuda.mem_get_info()[0]
    assert 120 * MB <= held <= 150 * MB, held / MB  # the driver maps memory in pieces of 2 MB and more


def test_a_larger_window_that_cannot_be_had_leaves_the_smaller():
    sc = scenes.cornell_spheres(width=16, height=16, depth=3, n_lon=24, n_lat=25)
    scene = jr.Scene(sc)
    states = []
    for fail in (False, True):
        ch = jr.Chains(scene, sc.width, sc.height, sc.depth, 3000, seed=2)
        ch.advance(40)
        if fail:
            jr.lib().jr_debug_fail_alloc(0)
        try:
            launches = ch.advance_timed(200)["path"]["launches"]
        finally:
            jr.lib().jr_debug_fail_alloc(-1)
        assert launches == (4 if fail else 1)  # windows of 64 steps, or one of 256
        states.append(ch.get_state())
    assert np.array_equal(states[0][0], states[1][0]) and np.array_equal(states[0][1], states[1][1])

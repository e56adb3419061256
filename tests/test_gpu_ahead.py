"""Look-ahead execution (the auto mode's choice where few steps are local)
against the megakernel and the wavefront on the same streams."""
import numpy as np
import pytest

from paper_2409_07148_gb300 import jr, scenes

pytestmark = pytest.mark.gpu

SCENES = {
    "box": lambda: scenes.cornell(width=32, height=32, depth=3),          # 24 triangles: one warp per chain settles
    "spheres": lambda: scenes.cornell_spheres(width=64, height=64, depth=5, n_lon=40, n_lat=41),
    "flat": lambda: scenes.cornell(width=8, height=8, depth=0),           # D = 2: no bounce, one Philox block, half used
    "empty": lambda: scenes.empty(),
}


def _run(sc, scene, n, mode, advances, flags, c_tilde):
    ch = jr.Chains(scene, sc.width, sc.height, sc.depth, n, seed=17, flags=flags, c_tilde=c_tilde, chain_offset=5)
    ch.set_execution(mode)
    for k in advances:
        ch.advance(k)
    return ch.get_state(), ch.stats(), ch.accumulator()


# 1 chain; 256: the latency case, over several calls; 4000: full warps of chains; 5000 and 20000: lanes of
# a warp at different steps; 1100000: windows of 15 steps, so a ragged last one and states carried over
@pytest.mark.parametrize("name,n,advances,other", [
    ("box", 1, [3, 70], "warp"), ("box", 256, [2, 33, 100], "warp"), ("box", 4000, [40], "mega"),
    ("flat", 1000, [50], "mega"), ("empty", 100, [39], "mega"), ("spheres", 1, [32], "mega"),
    ("spheres", 5000, [1, 2, 40], "mega"), ("spheres", 20000, [17], "mega"), ("spheres", 1100000, [20], "wave"),
])
@pytest.mark.parametrize("flags,c_tilde", [(0, 1.0), (jr.JR_FLAG_RAO_BLACKWELL, 0.3)])
def test_ahead_equals_the_other_modes(name, n, advances, other, flags, c_tilde):
    sc = SCENES[name]()
    scene = jr.Scene(sc)
    (xa, fa), sa, aa = _run(sc, scene, n, "auto", advances, flags, c_tilde)
    (xb, fb), sb, ab = _run(sc, scene, n, other, advances, flags, c_tilde)
    # the same device functions on the same draws: chains part only where a rounding that the
    # compiler places differently decides a tie
    same = np.all(xa == xb, axis=0)
    assert np.mean(~same) <= 1e-4
    assert np.allclose(fa[:, same], fb[:, same], rtol=1e-5, atol=0)
    steps = n * sum(advances)
    assert sa["regenerations"] + sa["local_steps"] == steps == sb["regenerations"] + sb["local_steps"]
    for key in ("regenerations", "local_steps", "accepted"):
        assert abs(sa[key] - sb[key]) <= 1e-5 * steps
    assert sa["status_word"] == sb["status_word"] == 0
    if np.all(same) and sa == sb:  # FP32 sums per pixel in another order
        assert np.allclose(aa, ab, rtol=1e-4, atol=1e-6 * np.abs(ab).max())


def test_ahead_reports_only_the_paths_a_chain_takes():
    """A budget that some rays exceed: the same status and the same chains as the
    wavefront, whatever was traced for nothing."""
    sc = SCENES["spheres"]()
    scene = jr.Scene(sc)
    out = []
    for mode in ("auto", "wave"):
        ch = jr.Chains(scene, sc.width, sc.height, sc.depth, 3000, seed=2)
        ch.set_execution(mode)
        ch.set_limits(node_visit_budget=12)
        ch.advance(40)
        out.append((ch.stats(check=False), *ch.get_state()))
    assert out[0][0]["status_word"] & jr.JR_STATUS_TRAVERSAL
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])
    assert np.allclose(out[0][2], out[1][2], rtol=1e-5, atol=0)


def test_ahead_without_memory_falls_back():
    sc = SCENES["spheres"]()
    scene = jr.Scene(sc)
    states = []
    for fail in (False, True):
        ch = jr.Chains(scene, sc.width, sc.height, sc.depth, 3000, seed=2)
        if fail:
            jr.lib().jr_debug_fail_alloc(0)
        try:
            ch.advance(33)
        finally:
            jr.lib().jr_debug_fail_alloc(-1)
        ch.advance(32)
        states.append(ch.get_state()[0])
    assert np.mean(np.all(states[0] == states[1], axis=0)) >= 1 - 1e-3


# several calls, so that the drifts stored at a window's end are used by the next; 1 chain; 3000: lanes
# at different steps, some with a drift to find first
@pytest.mark.parametrize("n,advances", [(1, [2, 40]), (3000, [3, 32, 33]), (40000, [5, 4])])
@pytest.mark.parametrize("c_tilde", [1.0, 0.05])
def test_ahead_mala_equals_the_megakernel(n, advances, c_tilde):
    sc = scenes.cornell_spheres(width=64, height=64, depth=4, n_lon=40, n_lat=41)
    scene = jr.Scene(sc)
    out = []
    for mode in ("auto", "mega"):
        ch = jr.Chains(scene, sc.width, sc.height, sc.depth, n, seed=23, flags=jr.JR_FLAG_MALA, sigma=0.02,
                       c_tilde=c_tilde)
        ch.set_execution(mode)
        for k in advances:
            ch.advance(k)
        out.append((ch.get_state(), ch.stats()))
    ((xa, fa), sa), ((xb, fb), sb) = out
    # a drift may differ in its last bit (the same function, compiled apart): 2 sigma 2^-23 in x
    same = np.all(np.abs(xa - xb) <= 1e-6, axis=0)
    assert np.mean(~same) <= 1e-3
    assert np.allclose(fa[:, same], fb[:, same], rtol=1e-4, atol=0)
    steps = n * sum(advances)
    assert sa["regenerations"] + sa["local_steps"] == steps
    for key in ("regenerations", "local_steps", "accepted"):
        assert abs(sa[key] - sb[key]) <= max(1, 1e-4 * steps)


def test_a_captured_advance_keeps_its_buffers():
    """A captured advance runs in the windows that an advance outside a capture left;
    a later, longer one leaves them where the graph has them; a captured advance too
    short for windows (2^18 chains: the wavefront's) still captures."""
    import torch
    sc = SCENES["spheres"]()
    scene = jr.Scene(sc)
    n = 1 << 18
    ends = []
    for capture in (False, True):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            ch = jr.Chains(scene, sc.width, sc.height, sc.depth, n, seed=17, stream=st)
            ch.advance(4, stream=st)
            st.synchronize()
            if not capture:
                ch.advance(4, stream=st)
                ch.advance(1, stream=st)
            else:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=st):
                    ch.advance(4, stream=st)
                    ch.advance(1, stream=st)
                g.replay()
            ch.advance(24, stream=st)
            st.synchronize()
            if capture:
                x, _ = ch.get_state(stream=st)
                g.replay()  # steps 4 to 8 once more, from the present states: in its own buffers
                st.synchronize()
                assert ch.stats()["status_word"] == 0
                ends.append(x)
            else:
                ends.append(ch.get_state(stream=st)[0])
    # windows of other lengths: other kernels for the tails, so ties as above
    assert np.mean(np.any(ends[0] != ends[1], axis=0)) <= 1e-4

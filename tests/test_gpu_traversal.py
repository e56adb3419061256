"""The traversal's watchdog variants: a launch checks only the limits that can
fire, and each variant gives the states of the one that checks both."""
import numpy as np
import pytest

from paper_2409_07148_gb300 import jr, scenes

pytestmark = pytest.mark.gpu


def _run(scene, sc, n, mode, limits, flags, steps=6):
    ch = jr.Chains(scene, sc.width, sc.height, sc.depth, n, seed=11, flags=flags, burn_in=0)
    ch.set_limits(*limits)
    ch.set_execution(mode)
    ch.advance(steps)
    x, fpu = ch.get_state()
    st = ch.stats()
    return x, fpu, st


# 1 and 33 chains: a lane alone and a warp plus one; 5000: many warps, ragged
@pytest.mark.parametrize("n", [1, 33, 5000])
@pytest.mark.parametrize("mode", ["wave", "mega"])
@pytest.mark.parametrize("flags", [0, jr.JR_FLAG_MH])
def test_check_variants_give_the_same_chains(n, mode, flags):
    sc = scenes.cornell_spheres(width=64, height=64, depth=6, n_lon=40, n_lat=41)
    scene = jr.Scene(sc)
    nodes = scene.info()["n_nodes"]
    assert 900 < nodes < 65536
    ref = _run(scene, sc, n, mode, (0, 0), flags)            # neither limit can fire
    visits = _run(scene, sc, n, mode, (nodes - 1, 0), flags)  # visits are counted, none runs out
    both = _run(scene, sc, n, mode, (0, 16), flags)           # every push is compared, none runs out
    for other in (visits, both):
        assert other[2] == ref[2]
        assert np.array_equal(other[0], ref[0])
        assert np.array_equal(other[1], ref[1])


@pytest.mark.parametrize("mode", ["wave", "mega"])
def test_budget_counted_once_per_round_equals_counted_per_visit(mode):
    """A budget that some rays exceed: the variant that compares once per round
    (stack limit out of reach) marks the same rays as the one that compares at
    every visit (a stack limit below the tree's bound, above what rays use)."""
    sc = scenes.cornell_spheres(width=64, height=64, depth=4, n_lon=40, n_lat=41)
    scene = jr.Scene(sc)
    out = []
    for limits in ((9, 0), (9, 16)):
        ch = jr.Chains(scene, sc.width, sc.height, sc.depth, 4096, seed=3, flags=jr.JR_FLAG_MH, burn_in=0)
        ch.set_limits(*limits)
        ch.set_execution(mode)
        ch.advance(4)
        st = ch.stats(check=False)
        assert st["status_word"] & jr.JR_STATUS_TRAVERSAL
        assert not st["status_word"] & jr.JR_STATUS_STACK
        out.append((st, *ch.get_state()))
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])
    assert np.array_equal(out[0][2], out[1][2])


# 1 and 7: a single warp; 1824 and 1825: one chain per warp on 152 SMs x 12 warps, and the first with
# two; 58369: full warps; 90001: more than the device holds at once
@pytest.mark.parametrize("n", [1, 7, 1824, 1825, 58369, 90001])
def test_spread_megakernel_equals_wavefront(n):
    """The same device functions on the same streams: the chains agree except
    where a rounding that the compiler places differently decides a tie."""
    sc = scenes.cornell_spheres(width=64, height=64, depth=5, n_lon=40, n_lat=41)
    scene = jr.Scene(sc)
    (xa, fa, sa), (xb, fb, sb) = (_run(scene, sc, n, mode, (0, 0), jr.JR_FLAG_MH, steps=3) for mode in ("mega", "wave"))
    same = np.all(xa == xb, axis=0)
    assert np.mean(~same) <= 1e-4
    assert np.allclose(fa[:, same], fb[:, same], rtol=1e-5, atol=0)
    assert abs(sa["accepted"] - sb["accepted"]) <= 1e-4 * n


# 70000 chains drain in the wavefront first and in the drain kernel afterwards, their shards in the
# drain kernel alone; 1 step: every tour that survives it is reported open; 4097: more than one launch
@pytest.mark.parametrize("max_steps", [1, 3, 4097])
@pytest.mark.parametrize("rao", [0, jr.JR_FLAG_RAO_BLACKWELL])
def test_drain_kernel_equals_wavefront_drain(max_steps, rao):
    sc = scenes.furnace(width=32, height=32, depth=3, albedo=0.6, emission=20.0)
    scene = jr.Scene(sc)

    def drain(offset, n):
        ch = jr.Chains(scene, sc.width, sc.height, sc.depth, n, seed=5, chain_offset=offset, flags=rao)
        ch.advance(2)
        left = jr.complete_tours(ch, max_steps)
        return left, ch.stats(), ch.accumulator()

    whole = drain(0, 70000)
    parts = [drain(0, 35000), drain(35000, 35000)]
    assert whole[0] == sum(p[0] for p in parts)
    assert (whole[0] > 0) == (max_steps < 4097)
    for key in ("regenerations", "local_steps", "accepted"):
        assert whole[1][key] == sum(p[1][key] for p in parts)
    assert whole[1]["steps_per_chain"] == max(p[1]["steps_per_chain"] for p in parts)
    acc = sum(p[2] for p in parts)
    # FP32 sums of up to a few thousand positive terms per pixel in another order
    assert np.allclose(whole[2], acc, rtol=1e-4, atol=0)


# 2^19 + 77 samples go to persistent warps, and a Phong scene's lit samples are listed (a
# ragged last block); calls below 2^17 samples take one thread per path.  FP64 sums
# of one pixel in another order: 2^20 additions at most, each 2^-53 relative, all
# terms of one sign: 1.2e-10.
@pytest.mark.parametrize("phong", [True, False])
def test_render_in_one_call_equals_split_calls(phong):
    if phong:
        sc = scenes.cornell_spheres(width=32, height=32, depth=6, n_lon=40, n_lat=41)
    else:
        sc = scenes.cornell(width=32, height=32, depth=6)
    scene = jr.Scene(sc)
    n, first = (1 << 19) + 77, (1 << 32) - 1000
    whole = jr.render_pt(scene, sc.width, sc.height, sc.depth, n, seed=5, sample_begin=first)
    parts = 0
    for a in range(0, n, 130_001):
        b = min(a + 130_001, n)
        parts = parts + jr.render_pt(scene, sc.width, sc.height, sc.depth, b - a, seed=5, sample_begin=first + a)
    assert whole[..., :3].sum() > 0
    np.testing.assert_allclose(whole[..., :3].cpu(), parts[..., :3].cpu(), rtol=1.2e-10, atol=0)


# 609 and 19 457 chains: one more than four warps per SM hold with one and with 32 chains each
# (152 SMs); the last 100 alone go one to a warp.  The same kernel on the same draws: equal.
@pytest.mark.parametrize("n", [609, 19457])
@pytest.mark.parametrize("name", ["cornell", "cornell_spheres"])
def test_mala_chains_do_not_depend_on_their_warps(n, name):
    sc = scenes.cornell(width=32, height=32, depth=3) if name == "cornell" else \
        scenes.cornell_spheres(width=32, height=32, depth=3, n_lon=40, n_lat=41)
    scene = jr.Scene(sc)
    x = []
    for chains, first in ((n, 0), (100, n - 100)):
        ch = jr.Chains(scene, sc.width, sc.height, sc.depth, chains, seed=3, flags=jr.JR_FLAG_MALA, chain_offset=first)
        ch.set_execution("mega")
        ch.advance(5)
        assert ch.stats()["status_word"] == 0
        x.append(ch.get_state())
    assert np.array_equal(x[0][0][:, -100:], x[1][0])
    assert np.array_equal(x[0][1][:, -100:], x[1][1])

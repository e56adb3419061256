"""Which advances run in look-ahead windows: the answer depends on the chain set's own parameters and
the number of steps, not on the states that the chains happen to hold."""
import pytest

from paper_2409_07148_gb300 import jr, scenes

pytestmark = pytest.mark.gpu

SCENES = {
    "box": lambda: scenes.cornell(width=64, height=64, depth=3),
    "caustic": lambda: scenes.caustic_slit(width=64, height=64, depth=10, n_lon=40, n_lat=41),
}


def _looks_ahead(ch, steps):
    """Path launches of one advance: one per window where it looks ahead, none in the
    megakernel and the warp mode, one per step in the wavefront."""
    launches = ch.advance_timed(steps)["path"]["launches"]
    assert launches in (0, steps) or launches < steps
    return 0 < launches < steps


# 256 and 3000 chains: states of the jump chain hold several times the p of samples of mu
@pytest.mark.parametrize("name,n,flags", [("box", 256, 0), ("caustic", 3000, 0), ("caustic", 3000, jr.JR_FLAG_MALA)])
@pytest.mark.parametrize("before", [0, 10, 31])
def test_earlier_short_advances_do_not_decide(name, n, flags, before):
    sc = SCENES[name]()
    scene = jr.Scene(sc)
    kw = dict(seed=4, flags=flags)
    ch = jr.Chains(scene, sc.width, sc.height, sc.depth, n, **kw)
    for _ in range(before):
        ch.advance(1)
    restored = jr.Chains(scene, sc.width, sc.height, sc.depth, n, **kw)
    restored.set_state(*ch.get_state())
    restored.set_counters(ch.stats(), ch.accumulator())
    assert _looks_ahead(ch, 100)
    assert _looks_ahead(restored, 100)


@pytest.mark.parametrize("n", [256, 3000])
def test_many_local_steps_do_not_look_ahead(n):
    """c~ = 0.02: about nine steps in ten are local in the box."""
    sc = SCENES["box"]()
    ch = jr.Chains(jr.Scene(sc), sc.width, sc.height, sc.depth, n, seed=4, c_tilde=0.02)
    assert not _looks_ahead(ch, 100)
    assert not _looks_ahead(ch, 100)


# a share of local steps of about 0.2 (c~ = 0.65): 256 and 608 chains are settled by blocks, 609 and 2000 by a
# warp each (152 SMs), where it takes more steps for a window to pay
@pytest.mark.parametrize("n,steps,expected", [(256, 32, True), (608, 32, True), (609, 32, False), (2000, 64, False),
                                              (609, 96, True), (2000, 96, True)])
def test_few_steps_of_a_warp_per_chain(n, steps, expected):
    sc = SCENES["box"]()
    ch = jr.Chains(jr.Scene(sc), sc.width, sc.height, sc.depth, n, seed=4, c_tilde=0.65)
    assert _looks_ahead(ch, steps) == expected
    assert _looks_ahead(ch, 200)  # asked again by every call

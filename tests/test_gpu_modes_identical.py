"""A chain's states do not depend on the kernel that runs its steps: every execution mode, and
any split of the steps into calls, gives the same bits, so a checkpoint restored into a fresh
chain set continues bit-identically although the auto mode picks its kernels by the call."""
import numpy as np
import pytest

from paper_2409_07148_gb300 import jr, scenes

pytestmark = pytest.mark.gpu

SCENES = {  # every material: Lambert, modified Phong, dielectric; small and large triangle counts
    "box": lambda: scenes.cornell(width=64, height=64, depth=3),
    "spheres": lambda: scenes.cornell_spheres(width=64, height=64, depth=8, n_lon=40, n_lat=41),
    "caustic": lambda: scenes.caustic_slit(width=64, height=64, depth=10, n_lon=40, n_lat=41),
    "glass": lambda: scenes.glass_furnace(width=32, height=32, depth=6),
    "terrain": lambda: scenes.terrain(width=64, height=64, depth=12, n_grid=60),
}


def _set(scene, sc, n, **kw):
    return jr.Chains(scene, sc.width, sc.height, sc.depth, n, seed=29, **kw)


def _same(a, b):
    (xa, fa), (xb, fb) = a.get_state(), b.get_state()
    assert np.array_equal(xa, xb) and np.array_equal(fa, fb), (np.any(xa != xb, axis=0).sum(), np.any(fa != fb, axis=0).sum())
    sa, sb = a.stats(), b.stats()
    # p_sum_large is a sum of doubles in no fixed order
    assert {k: v for k, v in sa.items() if k != "p_sum_large"} == {k: v for k, v in sb.items() if k != "p_sum_large"}


# 300 chains: windows settled a block per chain where the scene allows it; 3000 and 70000: by the tails;
# 300000: the wavefront's range.  c~ = 0.1: many lit states, whose F a last bit would show in.
@pytest.mark.parametrize("name", list(SCENES))
@pytest.mark.parametrize("n,steps", [(300, 120), (3000, 96), (70000, 48), (300000, 24)])
def test_modes_and_splits_are_bit_identical(name, n, steps):
    sc = SCENES[name]()
    scene = jr.Scene(sc)
    mega = _set(scene, sc, n, c_tilde=0.1)
    mega.set_execution("mega")
    mega.advance(steps)
    wave = _set(scene, sc, n, c_tilde=0.1)
    wave.set_execution("wave")
    wave.advance(steps)
    _same(wave, mega)
    auto = _set(scene, sc, n, c_tilde=0.1)
    auto.advance(steps)
    _same(auto, mega)
    first = _set(scene, sc, n, c_tilde=0.1)
    first.advance(steps // 3)
    rest = _set(scene, sc, n, c_tilde=0.1)  # the checkpoint
    rest.set_state(*first.get_state())
    rest.set_counters(first.stats(), first.accumulator())
    rest.advance(steps - steps // 3)
    _same(rest, mega)


@pytest.mark.parametrize("name", ["spheres", "caustic"])
def test_mh_modes_are_bit_identical(name):
    sc = SCENES[name]()
    scene = jr.Scene(sc)
    out = []
    for mode in ("mega", "wave"):
        ch = _set(scene, sc, 300000, flags=jr.JR_FLAG_MH, burn_in=0)
        ch.set_execution(mode)
        ch.advance(12)
        out.append(ch)
    _same(*out)


@pytest.mark.parametrize("name", ["spheres", "caustic", "glass"])
@pytest.mark.parametrize("n,steps", [(3000, 96), (40000, 24)])
def test_mala_splits_are_bit_identical(name, n, steps):
    sc = SCENES[name]()
    scene = jr.Scene(sc)
    kw = dict(flags=jr.JR_FLAG_MALA, sigma=0.02, c_tilde=0.1)
    mega = _set(scene, sc, n, **kw)
    mega.set_execution("mega")
    mega.advance(steps)
    auto = _set(scene, sc, n, **kw)
    auto.advance(steps)
    _same(auto, mega)
    first = _set(scene, sc, n, **kw)
    first.advance(steps // 3)
    rest = _set(scene, sc, n, **kw)
    rest.set_state(*first.get_state())
    rest.set_counters(first.stats(), first.accumulator())
    rest.advance(steps - steps // 3)
    _same(rest, mega)


# the batched wavefront and the batch megakernel, every material, over sets of uneven size
@pytest.mark.parametrize("block", [0, 64])
@pytest.mark.parametrize("flags", [0, jr.JR_FLAG_MH])
def test_batches_are_bit_identical(block, flags):
    scs = [SCENES[name]() for name in ("box", "spheres", "caustic", "glass")]
    alone, together = [], []
    for sc, n in zip(scs, (100, 3001, 20000, 700)):
        scene = jr.Scene(sc)
        for sets in (alone, together):
            sets.append(_set(scene, sc, n, c_tilde=0.1, flags=flags, burn_in=0))
    batch = jr.Batch(together)
    batch.set_block(block)
    batch.advance(12)
    for a, b in zip(alone, together):
        a.set_execution("mega")
        a.advance(12)
        _same(b, a)

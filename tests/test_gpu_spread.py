"""How many chains a warp of the megakernels holds does not change them: sizes on both sides of every
line of that rule, against the last 100 chains in a set of their own (one or two to a warp)."""
import numpy as np
import pytest

from paper_2409_07148_gb300 import jr, scenes

pytestmark = pytest.mark.gpu


def _alone_and_together(sc, n, **kw):
    scene = jr.Scene(sc)
    out = []
    for chains, first in ((n, 0), (100, n - 100)):
        ch = jr.Chains(scene, sc.width, sc.height, sc.depth, chains, seed=3, chain_offset=first, **kw)
        ch.set_execution("mega")
        ch.advance(4)
        assert ch.stats()["status_word"] == 0
        out.append(ch.get_state())
    (x, f), (xa, fa) = out
    assert np.array_equal(x[:, -100:], xa) and np.array_equal(f[:, -100:], fa)


# MALA on 152 SMs: D = 24 has 4 warps per SM (608, 609 chains: one and two per warp; 19456, 19457: 32 and full
# warps), D = 26 has 3 (456, 457; 14592, 14593); 58368, 58369: the last size that asks for its share of L1
@pytest.mark.parametrize("depth,n", [(11, 608), (11, 609), (11, 19456), (11, 19457), (12, 456), (12, 457),
                                     (12, 14592), (12, 14593), (15, 58368), (15, 58369), (0, 58369)])
@pytest.mark.parametrize("flags", [jr.JR_FLAG_MALA, jr.JR_FLAG_MALA | jr.JR_FLAG_MH])
def test_mala_chains_do_not_depend_on_their_warps(depth, n, flags):
    sc = scenes.cornell_spheres(width=32, height=32, depth=depth, n_lon=24, n_lat=25)
    _alone_and_together(sc, n, flags=flags, sigma=0.02, burn_in=0)


# 8 warps per SM up to 128 triangles, 12 above (152 SMs): the sizes at which a warp takes one chain more, and the
# largest that is spread at all
@pytest.mark.parametrize("name,n", [("box", 1216), ("box", 1217), ("box", 38913), ("box", 77824), ("box", 77825),
                                    ("spheres", 1824), ("spheres", 1825), ("spheres", 58369)])
@pytest.mark.parametrize("flags", [0, jr.JR_FLAG_MH])
def test_chains_do_not_depend_on_their_warps(name, n, flags):
    sc = scenes.cornell(width=32, height=32, depth=4) if name == "box" else \
        scenes.cornell_spheres(width=32, height=32, depth=4, n_lon=24, n_lat=25)
    _alone_and_together(sc, n, flags=flags, burn_in=0)

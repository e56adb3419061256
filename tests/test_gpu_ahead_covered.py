"""Look-ahead against the other modes, where it is known to run: the launches show it, with and without
Rao-Blackwellised splats, on every kernel that settles a window, and the image is always compared."""
import numpy as np
import pytest

from paper_2409_07148_gb300 import jr, scenes

pytestmark = pytest.mark.gpu

RAO = jr.JR_FLAG_RAO_BLACKWELL


def _advance(scene, sc, n, mode, advances, **kw):
    ch = jr.Chains(scene, sc.width, sc.height, sc.depth, n, seed=31, chain_offset=3, **kw)
    ch.set_execution(mode)
    launches = [ch.advance_timed(k)["path"]["launches"] for k in advances]
    return ch.get_state(), ch.stats(), ch.accumulator(), launches


# On 152 SMs the box's windows are settled three steps a round by a block per chain up to 304 chains, two up to
# 608, and by a warp per chain above; c~ = 1 and 0.7 give shares of local steps of about 0.14 and 0.19.  Spheres: the
# queued chains by blocks (3000), by the tail kernel (100000), and beside the next window's paths (300000: windows
# of 27 steps).
@pytest.mark.parametrize("name,n,advances,other,c_tilde", [
    ("box", 256, [3, 33, 64], "warp", 1.0), ("box", 256, [40], "warp", 0.7), ("box", 500, [3, 40], "warp", 1.0),
    ("box", 2000, [100, 96], "warp", 0.7), ("spheres", 3000, [2, 40], "mega", 0.05),
    ("spheres", 100000, [9, 16], "mega", 0.05), ("spheres", 300000, [60], "wave", 0.05),
])
@pytest.mark.parametrize("flags", [0, RAO])
def test_windows_equal_the_other_modes(name, n, advances, other, c_tilde, flags):
    sc = scenes.cornell(width=32, height=32, depth=3) if name == "box" else \
        scenes.cornell_spheres(width=64, height=64, depth=5, n_lon=40, n_lat=41)
    scene = jr.Scene(sc)
    kw = dict(flags=flags, c_tilde=c_tilde)
    (xa, fa), sa, aa, la = _advance(scene, sc, n, "auto", advances, **kw)
    (xb, fb), sb, ab, _ = _advance(scene, sc, n, other, advances, **kw)
    assert all(0 < m < k for m, k in zip(la, advances) if k >= 9), la  # windows, and not a launch per step
    assert sa["local_steps"] > 0.01 * n
    assert np.array_equal(xa, xb) and np.array_equal(fa, fb) and sa == sb
    # the same terms in another order, in FP32 per advance: at most n k of them, all of one sign, and half an
    # ulp each at worst grows like the square root: 2^-24 sqrt(n k / pixels) is below 1e-5
    assert np.allclose(aa, ab, rtol=1e-4, atol=0)
    assert np.isclose(aa.sum(), ab.sum(), rtol=1e-5)


@pytest.mark.parametrize("n,advances,c_tilde", [(3000, [32, 40], 1.0), (3000, [40], 0.1), (40000, [6, 4], 0.1)])
def test_mala_windows_equal_the_megakernel(n, advances, c_tilde):
    sc = scenes.cornell_spheres(width=64, height=64, depth=4, n_lon=40, n_lat=41)
    scene = jr.Scene(sc)
    kw = dict(flags=jr.JR_FLAG_MALA, sigma=0.02, c_tilde=c_tilde)
    (xa, fa), sa, aa, la = _advance(scene, sc, n, "auto", advances, **kw)
    (xb, fb), sb, ab, _ = _advance(scene, sc, n, "mega", advances, **kw)
    assert all(0 < m < k for m, k in zip(la, advances)), la
    assert np.array_equal(xa, xb) and np.array_equal(fa, fb) and sa == sb
    assert np.allclose(aa, ab, rtol=1e-4, atol=0)

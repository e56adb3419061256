"""Path tracing's two kernels (one thread per path, persistent warps): the same sums on every material,
and no device memory taken by a call."""
import ctypes

import numpy as np
import pytest

from paper_2409_07148_gb300 import jr, scenes

pytestmark = pytest.mark.gpu

SCENES = {  # Phong and Lambert, more and fewer than 128 triangles (the rules differ)
    "spheres": lambda: scenes.cornell_spheres(width=32, height=32, depth=6, n_lon=40, n_lat=41),
    "boxes": lambda: scenes.random_boxes(3, 100, 32, 32, 6),
    "box": lambda: scenes.cornell(width=32, height=32, depth=4),
}


# both sides of the lines (163 840 samples; 262 144 below 129 triangles) and an odd count above; the parts are
# below either.  FP64 sums of one pixel in another order: at most 2^19 additions, each 2^-53 relative, all terms
# of one sign: 6e-11.
@pytest.mark.parametrize("name", list(SCENES))
@pytest.mark.parametrize("n", [163839, 163840, 262143, 262144, 300001])
def test_persistent_paths_equal_one_thread_per_path(name, n):
    sc = SCENES[name]()
    scene = jr.Scene(sc)
    first = (1 << 32) - 1000
    whole = jr.render_pt(scene, sc.width, sc.height, sc.depth, n, seed=7, sample_begin=first)
    parts = 0
    for a in range(0, n, 100_003):
        m = min(100_003, n - a)
        parts = parts + jr.render_pt(scene, sc.width, sc.height, sc.depth, m, seed=7, sample_begin=first + a)
    assert whole[..., :3].sum() > 0
    np.testing.assert_allclose(whole[..., :3].cpu(), parts[..., :3].cpu(), rtol=6e-11, atol=0)


def test_a_render_takes_no_device_memory():
    """No allocation from the device's stream-ordered pool either: it gives its memory
    back at every synchronisation, so a call would pay for the mapping each time."""
    import torch
    sc = SCENES["spheres"]()
    scene = jr.Scene(sc)
    accum = torch.zeros((sc.height, sc.width, 4), dtype=torch.float64, device="cuda")
    jr.render_pt(scene, sc.width, sc.height, sc.depth, 1000, accum=accum)  # loads the kernels
    torch.cuda.synchronize()
    cuda = ctypes.CDLL("libcuda.so.1")
    pool, high = ctypes.c_void_p(), ctypes.c_uint64(0)
    assert cuda.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    used_mem_high = 8  # CU_MEMPOOL_ATTR_USED_MEM_HIGH
    assert cuda.cuMemPoolSetAttribute(pool, used_mem_high, ctypes.byref(high)) == 0  # reset
    assert cuda.cuMemPoolGetAttribute(pool, used_mem_high, ctypes.byref(high)) == 0
    before = high.value
    jr.render_pt(scene, sc.width, sc.height, sc.depth, 1 << 20, accum=accum)
    torch.cuda.synchronize()
    assert cuda.cuMemPoolGetAttribute(pool, used_mem_high, ctypes.byref(high)) == 0
    assert high.value == before

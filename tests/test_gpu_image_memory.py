"""Device memory of a handle's images, per voxel of all levels: R, T and the pass's copy of T 4 bytes each, 16 for
R's normalized gradient field where a pass reads it."""
import numpy as np
import pytest

from synth import random_image

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def taken(dims, **kw):
    """Bytes that set_images takes, less the scratch that does not depend on the image type (seen as a difference)."""
    import paper_1812_06765_gb300 as reg
    R = torch.from_numpy(random_image(dims, 7)).cuda()
    r = reg.Registration(reg.make_config(levels=1, autotune=False, **kw))
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    r.set_images(R, R, (1.0, 1.0, 1.0))
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    r.close()
    return used


def test_bf16_takes_no_more_than_fp32():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dims, page = (192, 160, 128), 4 << 20   # the driver hands out pages of 2 MB
    nv = int(np.prod(dims))
    taken(dims)                             # loads the kernels
    full = taken(dims)
    assert taken(dims, image_dtype="bf16") <= full + page
    # the passes that form the curvature (fused_tz = -1, as in batches) read no field: 12 bytes a voxel
    for dtype in ("f32", "bf16"):
        assert taken(dims, image_dtype=dtype, fused_tz=-1) <= full - 16 * nv + page

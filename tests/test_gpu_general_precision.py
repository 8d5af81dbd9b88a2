"""D on grids of other ratios than 2 is as close to 64 bits as the multi-pass kernels bring it."""
import numpy as np
import pytest

from synth import random_field, random_image

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tau", [0.1, 0.05, 0.3])
def test_d_has_no_bias(orc, tau):
    """psi = num / na2 takes a dozen FP32 roundings (2^-24 = 6e-8 each, to nearest) and an approximate
    reciprocal of mean error 4e-9: over 10^5 voxels they average out, and what stays is the mean of the
    roundings that all voxels share.  1.5e-8, a quarter of one rounding, leaves room for none of those."""
    import paper_1812_06765_gb300 as reg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tau = float(np.float32(tau))   # the FP32 value the kernels take: its own rounding is no error of theirs
    dims, h = (61, 57, 49), (1.0, 1.0, 1.0)
    err = []
    for seed in range(4):
        R, T = random_image(dims, 60 + seed), random_image(dims, 70 + seed)
        r = reg.Registration(reg.make_config(levels=1, tau=tau, alpha=1.0)).set_images(R, T, h)
        u = random_field(r.level_info(0)["nodes"], 80 + seed, 1.5)
        D = r.eval(torch.from_numpy(u).cuda())[1]
        Do = orc.objective(dims, h, R, T, r.level_info(0)["nodes"], u, tau, tau, 1.0)[1]
        err.append((D - Do) / Do)
        r.close()
    assert abs(np.mean(err)) <= 1.5e-8, err

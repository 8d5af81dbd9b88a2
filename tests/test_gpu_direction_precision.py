"""The direction of given pairs keeps the accuracy of short FP32 sums."""
import numpy as np
import pytest

from synth import random_image
from tests.test_gpu_direction import two_loop

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def combined(S, Y, g):
    """The direction with dots and coefficients in 64 bits, combined in FP32 in the kernel's order: what is left
    of the error when the sums have none."""
    Sd, Yd, gd = S.double(), Y.double(), g.double()
    c = len(S)
    SY, YY = Sd @ Yd.T, Yd @ Yd.T
    gam = SY[-1, -1] / YY[-1, -1]
    q = torch.linalg.solve_triangular(torch.triu(SY), (Sd @ gd)[:, None], upper=True)[:, 0]
    rhs = torch.diag(SY) * q + gam * (YY @ q - Yd @ gd)
    w = torch.linalg.solve_triangular(torch.triu(SY).T, rhs[:, None], upper=False)[:, 0]
    x = (-gam).float() * g
    for j in range(c):   # fma: products of two FP32 numbers are exact in 64 bits
        t = ((gam * q[j]).float().double() * Yd[j] + x.double()).float()
        x = ((-w[j]).float().double() * Sd[j] + t.double()).float()
    return x


# The sums of few unknowns: a block's FP32 partial of one product per thread carries about 2.5e-8, and
# the partials' errors average over the blocks.  Simulated over 32 draws the whole error is 1.29, 1.13
# and 1.05 times that of exact sums at these sizes, with 4 products per thread on a quarter of the
# blocks 1.89, 1.46 and 1.16 times: the bars lie between.
@pytest.mark.parametrize("n,count,bar", [(1023, 1, 1.55), (768, 3, 1.28), (2187, 5, 1.1)])
def test_short_sums(n, count, bar):
    import paper_1812_06765_gb300 as reg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = reg.Registration(reg.make_config(levels=1, mem=8)).set_images(
        random_image((16, 16, 16), 1), random_image((16, 16, 16), 2), (1.0, 1.0, 1.0))
    err, floor = [], []
    for seed in range(64):
        rng = np.random.default_rng([seed, n])
        S = rng.standard_normal((count, n)).astype(np.float32)
        Y = (S * rng.uniform(0.5, 3.0, n) + 0.05 * rng.standard_normal((count, n))).astype(np.float32)
        S, Y = torch.from_numpy(S).cuda(), torch.from_numpy(Y).cuda()
        g = torch.from_numpy(rng.standard_normal(n).astype(np.float32)).cuda()
        ref = two_loop(S, Y, g, 1.0)
        err.append(float((r.lbfgs_direction(S, Y, g).double() - ref).norm() / ref.norm()))
        floor.append(float((combined(S, Y, g).double() - ref).norm() / ref.norm()))
    r.close()
    assert np.sqrt(np.mean(np.square(err))) <= bar * np.sqrt(np.mean(np.square(floor)))


# where the split of the work changes (a chunk of 1024 per SM), and sums of hundreds of terms per thread
@pytest.mark.parametrize("n", [152 * 1024 - 1, 152 * 1024, 152 * 1024 + 1, 3 * 129 ** 3])
@pytest.mark.parametrize("count", [5, 8])
def test_long_sums(n, count):
    import paper_1812_06765_gb300 as reg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = reg.Registration(reg.make_config(levels=1, mem=8)).set_images(
        random_image((16, 16, 16), 1), random_image((16, 16, 16), 2), (1.0, 1.0, 1.0))
    gen = torch.Generator(device="cuda").manual_seed(n + count)
    S = torch.randn((count, n), generator=gen, device="cuda")
    Y = S * (0.5 + 2.5 * torch.rand(n, generator=gen, device="cuda"))
    g = torch.randn(n, generator=gen, device="cuda")
    ref = two_loop(S, Y, g, 1.0)
    # the FP32 combination, 2 count + 1 terms: half a dozen to a dozen roundings of 6e-8 a value
    assert float((r.lbfgs_direction(S, Y, g).double() - ref).norm()) <= 5e-7 * float(ref.norm())
    r.close()

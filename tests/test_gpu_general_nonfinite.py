"""The general-ratio objective pass where values are not finite or out of range: as the multi-pass
kernels (eval_impl = 1), which treat a sample with an unusable displacement as outside the image and
let a voxel reach only the nodes on which it has a weight."""
import numpy as np
import pytest

from synth import random_field, random_image
from tests.helpers import GRAD_RTOL, J_RTOL, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SPACING = (1.0, 1.3, 0.8)


def both(dims, nodes, R, T, u):
    """D and the gradient of the general pass and of the multi-pass kernels (alpha small, so that D's part shows)."""
    import paper_1812_06765_gb300 as reg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = []
    for impl in (0, 1):
        cfg = reg.make_config(levels=1, tau=0.06, rho=0.04, alpha=1e-3, node_dims=[nodes], eval_impl=impl)
        r = reg.Registration(cfg).set_images(R, T, SPACING)
        J, D, S, g = r.eval(torch.from_numpy(u).cuda())
        out.append((D, g.cpu().numpy()))
        r.close()
    return out


def assert_same(a, b):
    (D0, g0), (D1, g1) = a, b
    assert np.isfinite(D0) and np.isfinite(D1)
    assert abs(D0 - D1) <= J_RTOL * abs(D1)
    assert np.array_equal(np.isfinite(g0), np.isfinite(g1))
    ok = np.isfinite(g1)
    assert rel_l2(g0[ok], g1[ok]) <= GRAD_RTOL


# a node on an edge of the grid, which no curvature stencil reads: five fixed taps, run-time windows;
# 31 x 21 x 17 on 13 x 9 x 7: the voxel planes through the node planes 6 (x) and 3 (z) have no weight on the next ones
FORMS = [((29, 13, 10), (15, 7, 6)), ((64, 48, 40), (17, 13, 11)), ((31, 21, 17), (13, 9, 7))]


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3e6, -1.5e6])
@pytest.mark.parametrize("dims,nodes", FORMS)
def test_unusable_displacements_are_outside_the_image(dims, nodes, value):
    R, T = random_image(dims, 51), random_image(dims, 52)
    for comp, (kx, ky, kz) in enumerate([(0, 0, nodes[2] // 2 + 1), (nodes[0] // 2 + 1, 0, 0), (0, nodes[1] // 2, 0)]):
        u = random_field(nodes, 53, 1.0).astype(np.float32)
        u[comp, kz, ky, kx] = value
        assert_same(*both(dims, nodes, R, T, u))


# T~ is not finite at voxels of an edge of the image, which no interior voxel's central difference
# reads (u = 0: a cell reaches from a voxel to the next ones, so the edges at 0 in two dimensions)
@pytest.mark.parametrize("value", [np.inf, np.nan])
@pytest.mark.parametrize("dims,nodes", FORMS)
def test_template_not_finite_off_the_interior(dims, nodes, value):
    R, T = random_image(dims, 54), random_image(dims, 55)
    mx, my, mz = dims
    for z, y, x in [(0, 0, mx // 2), (0, my // 2, 0), (mz // 2, 0, 0), (0, 0, 0)]:
        Tn = T.copy()
        Tn[z, y, x] = value
        assert_same(*both(dims, nodes, R, Tn, np.zeros((3,) + nodes[::-1], np.float32)))

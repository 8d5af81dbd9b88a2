"""Parity on the routes that the other tests leave out: node grids of fewer than 2 voxels per interval (the
multi-pass kernels by default), rows of an odd length and of 2 more than a multiple of 4 in volumes large
enough for several planes per thread, curvature blocks of 2 and 3 node planes, and images of other scales."""
import numpy as np
import pytest

from synth import random_field, random_image
from tests.helpers import J_RTOL, assert_parity, compare_eval

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

H = (1.0, 1.3, 0.8)


@pytest.fixture(scope="module")
def reg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_06765_gb300
    return paper_1812_06765_gb300


def check(reg, orc, dims, nodes=None, tau=0.06, rho=0.04, alpha=2.0, scale=1.0, amp=1.5, **kw):
    R, T = (random_image(dims, s) * np.float32(scale) for s in (31, 32))
    cfg = reg.make_config(levels=1, tau=tau * scale, rho=rho * scale, alpha=alpha,
                          node_dims=[nodes] if nodes else None, **kw)
    r = reg.Registration(cfg).set_images(R, T, H)
    if kw.get("image_dtype") == "bf16":
        R, T = (torch.from_numpy(x).bfloat16().float().numpy() for x in (R, T))
    u = random_field(r.level_info(0)["nodes"], 33, amp)
    e = compare_eval(r, orc, R, T, dims, H, u, tau * scale, rho * scale, alpha)
    r.close()
    assert e["eD"] <= J_RTOL and e["eS"] <= 1e-5, {k: v for k, v in e.items() if k not in ("g", "go")}
    assert_parity(e)
    return e


# every dimension dense, one of them just over the limit, more nodes than voxels
@pytest.mark.parametrize("dims,nodes", [((20, 18, 16), (15, 13, 12)), ((20, 20, 20), (12, 11, 11)),
                                        ((20, 20, 20), (11, 11, 12)), ((19, 21, 17), (30, 9, 25))])
def test_dense_grids_take_the_multi_pass_kernels(reg, orc, dims, nodes):
    a, b = check(reg, orc, dims, nodes), check(reg, orc, dims, nodes, eval_impl=1)
    np.testing.assert_array_equal(a["g"], b["g"])      # the same kernels, not another pass's rounding
    assert a["D"] == b["D"]


def test_grids_at_the_limit_take_the_general_pass(reg, orc):
    dims, nodes = (20, 20, 21), (11, 11, 11)
    a, b = check(reg, orc, dims, nodes), check(reg, orc, dims, nodes, eval_impl=1)
    assert not np.array_equal(a["g"], b["g"])


@pytest.mark.parametrize("nodes", [[(15, 13, 12), (6, 5, 5)], [(11, 10, 9), (8, 7, 7)]])
def test_dense_and_sparse_levels_in_one_solve(reg, orc, nodes):
    dims, h = (20, 18, 16), (1.2, 1.0, 1.5)
    R = random_image(dims, 41)
    T = np.roll(R, shift=(1, -1, 1), axis=(0, 1, 2))
    kw = dict(levels=2, tau=0.05, alpha=5.0, mem=4, max_iter=5, fixed_iters=True, node_dims=nodes + [nodes[-1]] * 6)
    r = reg.Registration(reg.make_config(**kw)).set_images(R, T, h)
    u, st = r.register(out="numpy")
    uo, sto = orc.register(dims, h, R, T, orc.make_config(**kw))
    r.close()
    assert st["iters"] == sto["iters"] == [5, 5]
    du = np.sqrt(((u.astype(np.float64) - uo) ** 2).sum(axis=0))
    assert du.mean() / min(h) <= 0.02
    for lv in range(2):   # the bars of the other solver tests: the same path, or one that an Armijo test branched
        tol = 1e-4 if st["evals"][lv] == sto["evals"][lv] else 1e-2
        assert abs(st["J"][lv] - sto["J"][lv]) <= tol * abs(sto["J"][lv])


# more than 2^20 voxels; rows of 1, 2 and 3 more than a multiple of 4, depths that 4 does not divide
@pytest.mark.parametrize("dims,kw", [((181, 109, 67), {}), ((183, 107, 70), {}), ((182, 106, 67), {}),
                                     ((182, 106, 66), {}), ((182, 106, 66), dict(image_dtype="bf16"))])
def test_large_volumes_with_unaligned_rows(reg, orc, dims, kw):
    check(reg, orc, dims, **kw)


# 2 and 3 node planes per curvature block, the last block with fewer (alpha large: the curvature's part shows)
@pytest.mark.parametrize("nodes", [(104, 103, 105), (118, 117, 116)])
def test_curvature_blocks_of_several_planes(reg, orc, nodes):
    check(reg, orc, (60, 52, 48), nodes, alpha=50.0, amp=1.0)


# NGF is the same for images, tau and rho times one factor; the field of R is formed in the kernel's own
# quotients; 80 x 72 x 64 is the smallest ratio-2 grid of the three that reads it
@pytest.mark.parametrize("scale", [2.0 ** -40, 2.0 ** 40])
@pytest.mark.parametrize("dims", [(80, 72, 64), (61, 37, 43)])
def test_scaled_images(reg, orc, dims, scale):
    a, b = check(reg, orc, dims, scale=scale), check(reg, orc, dims)
    assert abs(a["D"] - b["D"]) <= 1e-6 * b["D"]


@pytest.mark.parametrize("dims", [(80, 72, 64), (61, 37, 43)])
def test_flat_and_faint_regions_of_the_reference(reg, orc, dims):
    """Exactly flat blocks (a divisor of rho itself) and gradients down to 1e-20 of rho beside ordinary ones."""
    R, T = random_image(dims, 61), random_image(dims, 62)
    R[:, :, : dims[0] // 3] = 0.25
    R[:, : dims[1] // 3, dims[0] // 3:] *= np.float32(1e-20)
    r = reg.Registration(reg.make_config(levels=1, tau=0.06, rho=0.04, alpha=2.0)).set_images(R, T, H)
    u = random_field(r.level_info(0)["nodes"], 63, 1.0)
    e = compare_eval(r, orc, R, T, dims, H, u, 0.06, 0.04, 2.0)
    r.close()
    assert e["eD"] <= J_RTOL
    assert_parity(e)

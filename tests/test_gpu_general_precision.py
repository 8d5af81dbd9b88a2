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


@pytest.mark.parametrize("dims,nodes", [((361, 21, 19), None), ((361, 24, 20), (91, 7, 6)), ((25, 23, 721), None),
                                        ((21, 361, 18), (9, 145, 7))])
def test_small_weights_of_the_adjoint(dims, nodes):
    """P^T's weight on the node before a voxel just below a node: a single bright template voxel, u = 0,
    so that the voxels that the gradient sees share one index along the long axis, and the gradient at
    the two nodes around it has exactly the ratio of the two weights.  1 - (FP32 weight of the other
    node) is off by up to 3e-8 of weights of 1 / m; each side here is a dozen FP32 roundings: 2e-6."""
    import paper_1812_06765_gb300 as reg
    from paper_1812_06765_gb300 import _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nodes = nodes or tuple(m // 2 + 1 for m in dims)
    axis = int(np.argmax(dims))
    k0, w1 = _lib.reg_axis_tables(dims[axis], 1.0, nodes[axis])[:2]
    t = (np.arange(dims[axis]) + 0.5) * (nodes[axis] - 1) / dims[axis]
    low = 1.0 - (t - k0)                                        # the lower node's weight in 64 bits
    loss = np.abs((np.float32(1) - np.asarray(w1, np.float32)).astype(np.float64) - low) / low
    loss[:8] = loss[-8:] = 0
    i = int(np.argmax(loss))
    assert loss[i] > 4e-6                                       # the voxel where rounding the other weight shows most
    p = [m // 2 for m in dims]
    p[axis] = i
    R, T = random_image(dims, 90), np.zeros(dims[::-1], np.float32)
    T[p[2], p[1], p[0]] = 1.0
    r = reg.Registration(reg.make_config(levels=1, tau=0.06, alpha=1.0, node_dims=[nodes])).set_images(R, T, (1.0,) * 3)
    g = r.eval(torch.zeros((3,) + nodes[::-1], device="cuda"))[3].cpu().numpy().astype(np.float64)
    r.close()
    g = np.moveaxis(g[1 if axis == 0 else 0], 2 - axis, 0)      # a component across the axis, the axis first
    lo, hi = g[k0[i]], g[k0[i] + 1]
    j = np.unravel_index(np.argmax(np.abs(hi)), hi.shape)
    assert hi[j] != 0
    assert abs(lo[j] / hi[j] - low[i] / (1.0 - low[i])) <= 2e-6 * low[i] / (1.0 - low[i])


def test_tile_totals_of_d_are_not_rounded():
    """Ramps across each other: psi is the same FP32 number at every interior voxel, so D / (hbar / 2) over
    their count is that number again, up to the FP64 and double-float sums (2^-46, 1e-10 allows for 10^3
    of them); a tile total rounded to FP32 would leave up to 6e-8."""
    import paper_1812_06765_gb300 as reg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for dims in [(61, 57, 49), (85, 43, 131), (29, 13, 21)]:
        z, y, x = np.meshgrid(*[np.arange(m) for m in dims[::-1]], indexing="ij")
        R, T = (x / 64.0).astype(np.float32), (y / 128.0).astype(np.float32)
        r = reg.Registration(reg.make_config(levels=1, tau=0.07, rho=0.03, alpha=1.0)).set_images(R, T, (1.0,) * 3)
        D = r.eval(torch.zeros((3,) + tuple(m // 2 + 1 for m in dims[::-1]), device="cuda"))[1]
        r.close()
        psi = D / (0.5 * np.prod([m - 2 for m in dims]))
        assert abs(psi - float(np.float32(psi))) <= 1e-10 * psi, (dims, psi)

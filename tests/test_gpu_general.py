"""The general-ratio objective pass where its tiles, windows and segments can go wrong."""
import numpy as np
import pytest

from synth import random_field, random_image
from tests.helpers import J_RTOL, assert_parity, compare_eval

torch = pytest.importorskip("torch")

# (dims, node dims or None for the default rule)
FORMS = [
    ((5, 4, 7), None),                    # smallest odd grid
    ((28, 12, 9), None),                  # one exact tile, odd depth only
    ((29, 13, 10), None),                 # a tile column and row of one voxel
    ((57, 25, 31), None),                 # the same, odd in every dimension
    ((31, 25, 131), None),                # several z segments, segment edges inside node intervals
    ((64, 48, 40), (17, 13, 11)),         # ratio 4
    ((66, 50, 70), (23, 18, 25)),         # ratios just under and at 3
    ((90, 70, 64), (3, 3, 3)),            # intervals wider than a tile and longer than a segment
    ((60, 40, 32), (31, 11, 4)),          # ratios 2, 4 and 10.7
    ((61, 37, 43), (31, 5, 22)),          # 2.03, 9.25, 2.05
    ((31, 21, 17), (13, 9, 7)),           # 5 weights a node, but 6 voxels in its intervals (one on a node)
    ((41, 11, 25), (17, 5, 11)),          # the same, and exactly 2.5
]


def test_tables_keep_the_tile_bounds():
    """What the pass's fixed arrays rely on at 2 or more voxels per node interval: the intervals of
    32 and 28 (16 and 12) columns in a row, a plane advancing by one interval at most every other plane."""
    from paper_1812_06765_gb300 import _lib
    for m in list(range(4, 80)) + [181, 217, 255, 256, 511]:
        for n in {m // 2 + 1, max(3, m // 4 + 1), max(3, m // 3), 3}:
            if 2 * (n - 1) > m or n < 3:
                continue
            k0 = _lib.reg_axis_tables(m, 0.97, n)[0]
            step = np.diff(k0)
            assert step.min() >= 0 and step.max() <= 1 and not np.any((step[1:] == 1) & (step[:-1] == 1))
            for cols, bound in ((32, 16), (28, 14), (16, 8), (12, 6)):
                span = [k0[min(i + cols, m) - 1] - k0[i] for i in range(m)]
                assert max(span) <= bound, (m, n, cols)


@pytest.mark.gpu
@pytest.mark.parametrize("dims,nodes", FORMS)
def test_general_pass_parity(orc, dims, nodes):
    import paper_1812_06765_gb300 as reg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    h = (1.0, 1.3, 0.8)
    R, T = random_image(dims, 31), random_image(dims, 32)
    cfg = reg.make_config(levels=1, tau=0.06, rho=0.04, alpha=2.0, node_dims=[nodes] if nodes else None)
    r = reg.Registration(cfg).set_images(R, T, h)
    u = random_field(r.level_info(0)["nodes"], 33, 1.5)
    e = compare_eval(r, orc, R, T, dims, h, u, 0.06, 0.04, 2.0)
    assert e["eD"] <= J_RTOL and e["eS"] <= 1e-5, e
    assert_parity(e)
    r.close()


@pytest.mark.gpu
@pytest.mark.parametrize("image_dtype", ["f32", "bf16"])
@pytest.mark.parametrize("dims,nodes", [FORMS[3], FORMS[5]])
def test_general_pass_in_the_solver(orc, dims, nodes, image_dtype):
    """Trial points u + t dir: a fixed number of steps follows the oracle (images stay FP32 on these levels)."""
    import paper_1812_06765_gb300 as reg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    h = (1.2, 1.0, 1.5)
    R = random_image(dims, 41)
    T = np.roll(R, shift=(1, -1, 1), axis=(0, 1, 2))
    kw = dict(levels=1, tau=0.05, alpha=5.0, mem=4, max_iter=5, fixed_iters=True,
              node_dims=[nodes] * 8 if nodes else None)
    r = reg.Registration(reg.make_config(image_dtype=image_dtype, **kw)).set_images(R, T, h)
    u, st = r.register(out="numpy")
    uo, sto = orc.register(dims, h, R, T, orc.make_config(**kw))
    assert st["iters"] == sto["iters"] == [5]
    du = np.sqrt(((u.astype(np.float64) - uo) ** 2).sum(axis=0))
    assert du.mean() / min(h) <= 0.02
    tol = 1e-4 if st["evals"] == sto["evals"] else 1e-2
    assert abs(st["J"][0] - sto["J"][0]) <= tol * abs(sto["J"][0])
    r.close()

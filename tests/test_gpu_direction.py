"""The L-BFGS direction of given pairs at the sizes where its passes can go wrong."""
import numpy as np
import pytest

from synth import random_image

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def two_loop(S, Y, g, hmin):
    """-H g in 64 bits (Nocedal's recursion, H0 = s'y / y'y of the newest pair)."""
    S, Y, q = S.double(), Y.double(), g.double().clone()
    if len(S) == 0:
        return -q * (hmin / float(q.abs().max()))
    a = [0.0] * len(S)
    for i in reversed(range(len(S))):
        a[i] = (S[i] @ q) / (S[i] @ Y[i])
        q -= a[i] * Y[i]
    q *= (S[-1] @ Y[-1]) / (Y[-1] @ Y[-1])
    for i in range(len(S)):
        q += S[i] * (a[i] - (Y[i] @ q) / (S[i] @ Y[i]))
    return -q


# one element, one short chunk, the edges of a chunk of 1024, more chunks than blocks (2 per SM), odd row lengths
@pytest.mark.parametrize("n", [1, 5, 1023, 1024, 1025, 4099, 311 * 1024 + 7, 3 * 65 ** 3])
@pytest.mark.parametrize("count", [0, 1, 2, 5, 8])
def test_direction_matches_two_loop(n, count):
    import paper_1812_06765_gb300 as reg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = reg.Registration(reg.make_config(levels=1, mem=8)).set_images(
        random_image((16, 16, 16), 1), random_image((16, 16, 16), 2), (1.0, 1.0, 1.0))
    gen = torch.Generator(device="cuda").manual_seed(1000 * count + n)
    count_n = min(count, max(n // 2, 1))   # more pairs than unknowns would be dependent
    # rows of a larger array that starts one element late: 4-byte alignment only
    buf = torch.randn(2 * count_n * n + n + 1, generator=gen, device="cuda")[1:]
    S = buf[:count_n * n].view(count_n, n)[:0 if count == 0 else count_n]
    stiff = 0.5 + 2.5 * torch.rand(n, generator=gen, device="cuda")
    Y = buf[count_n * n:2 * count_n * n].view(count_n, n)
    Y.copy_(buf[:count_n * n].view(count_n, n) * stiff)
    Y = Y[:len(S)]
    g = buf[2 * count_n * n:2 * count_n * n + n]
    p = r.lbfgs_direction(S if count else None, Y if count else None, g)
    ref = two_loop(S, Y, g, min(r.level_info(0)["node_spacing"]))
    # FP32 sums of at most 2^10 terms per thread and the FP32 combination: 2e-5, the bar of the other
    # direction test; with few unknowns the recursion cancels, so the bar is on the scale of gamma g too
    scale = max(float(ref.norm()), float(g.norm()) / 3.0)
    assert float((p.double() - ref).norm()) <= 2e-5 * scale
    r.close()

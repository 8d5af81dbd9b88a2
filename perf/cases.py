"""What a user of the registration library has it do, as measurable cases.

Every case goes through the package's public entry points
(`Registration`, `RegObjective`, `register`, `register_batch`).  The kinds:

  eval       one objective + gradient evaluation at a displacement: the call that
             an outer optimiser, a validation script or the solver itself repeats
  autograd   the objective as a differentiable scalar, forward and backward
  images     a new pair of images into an existing handle (the next frame of a
             4D series): copies, pyramid, the per-level fields of the solver
  direction  one L-BFGS direction from stored pairs
  register   the whole one-call registration, handle included
  batch      several prepared pairs of uneven size registered together

Images are CT-like phantoms in [0, 1] (a body, organs, 20 HU of noise) and their
warped counterparts; displacements are smooth fields of several voxels with a
little unevenness, as the solver meets them on the way to the solution.  J, D
and S come back as FP32, the precision of the terms they sum.
"""
import math

import numpy as np
import torch

import paper_1812_06765_gb300 as reg

TAU, ALPHA = 0.1, 50.0     # edge parameter and curvature weight of the CT workloads
MEM = 5                    # L-BFGS memory


def listed():
    return [
        # the coarsest pyramid level of a small pair, and a thumbnail-sized problem: launches and latency
        dict(name="eval_32", kind="eval", dims="32x32x32", spacing="1.5x1.5x1.5", nodes="half", dtype="f32"),
        # a CT pair at 1.5 mm, the middle level of a larger one
        dict(name="eval_128", kind="eval", dims="128x128x128", spacing="1.5x1.5x1.5", nodes="half", dtype="f32"),
        # the headline size: a 256^3 CT pair at 1 mm
        dict(name="eval_256", kind="eval", dims="256x256x256", spacing="1.0x1.0x1.0", nodes="half", dtype="f32"),
        # half a full-resolution thorax: the largest volumes of the tests
        dict(name="eval_fullres", kind="eval", dims="512x512x256", spacing="0.75x0.75x0.75", nodes="half",
             dtype="f32"),
        # a lung 4D-CT pair with 16-bit image storage
        dict(name="eval_lung_bf16", kind="eval", dims="256x256x112", spacing="0.97x0.97x2.5", nodes="half",
             dtype="bf16"),
        # odd sizes in every dimension, as scanners and brain atlases give them
        dict(name="eval_odd", kind="eval", dims="181x217x181", spacing="1.0x1.0x1.0", nodes="half", dtype="f32"),
        # the lung pair on the paper's 4D-CT grid, a quarter of the image resolution
        dict(name="eval_quarter", kind="eval", dims="256x256x112", spacing="0.97x0.97x2.5", nodes="quarter",
             dtype="f32"),
        # the objective inside a PyTorch program: forward and backward, anisotropic voxels
        dict(name="autograd_96", kind="autograd", dims="96x80x72", spacing="1.2x1.2x2.0", nodes="half",
             dtype="f32"),
        # the next frame of a lung series into its handle
        dict(name="images_lung", kind="images", dims="256x256x112", spacing="0.97x0.97x2.5", levels=4),
        # one L-BFGS direction on the grid of a 128^3 pair, full memory
        dict(name="direction_65", kind="direction", nodes="65x65x65", count=5),
        # the README's call on a small CT pair, from the displacement of the frame before it,
        # with the few iterations of an interactive tool
        dict(name="register_64", kind="register", dims="64x64x64", spacing="2.0x2.0x2.0", levels=2, iters=4),
        # regions of interest of uneven size registered together, a few iterations per level
        dict(name="batch_6", kind="batch", levels=2, iters=2, spacing="1.5x1.5x1.5",
             sizes="48x48x48 64x64x64 80x80x64 64x64x64 96x96x96 80x80x80"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dims(rng, voxels, multiple=1, least=16):
    """Three sides of about `voxels` voxels in all, none more than about three times another."""
    f = [_log_uniform(rng, 0.6, 1.7) for _ in range(3)]
    s = (voxels / (f[0] * f[1] * f[2])) ** (1.0 / 3.0)
    return _text([max(least, multiple * int(round(s * a / multiple))) for a in f])


def _text(sizes):
    return "x".join(str(v) for v in sizes)


def _sizes(text):
    return [int(v) for v in text.split("x")]


def _mm(case):
    return [float(v) for v in case["spacing"].split("x")]


def _spacing(rng):
    h = round(rng.uniform(0.7, 2.0), 2)
    return _text([h, h, round(h * rng.choice([1.0, 1.0, 1.5, 2.5]), 3)])


def draw(rng):
    kind = rng.choice(["eval"] * 5 + ["autograd", "images", "direction", "register", "batch"])
    if kind in ("eval", "autograd"):
        form = rng.choice(["even", "even", "bf16", "odd", "quarter"])
        voxels = _log_uniform(rng, 24.0 ** 3, 3.5e7 if kind == "eval" else 4e6)
        return dict(kind=kind, dims=_dims(rng, voxels, 2 if form in ("even", "bf16") else 1), spacing=_spacing(rng),
                    nodes="quarter" if form == "quarter" else "half", dtype="bf16" if form == "bf16" else "f32")
    if kind == "images":
        voxels = _log_uniform(rng, 40.0 ** 3, 2e7)
        return dict(kind=kind, dims=_dims(rng, voxels, rng.choice([1, 8, 8]), 40), spacing=_spacing(rng),
                    levels=rng.randint(2, 4))
    if kind == "direction":
        return dict(kind=kind, nodes=_dims(rng, _log_uniform(rng, 9.0 ** 3, 129.0 ** 3), 1, 7), count=rng.randint(1, 8))
    if kind == "register":
        voxels = _log_uniform(rng, 32.0 ** 3, 80.0 ** 3)
        return dict(kind=kind, dims=_dims(rng, voxels, rng.choice([1, 4, 4, 4]), 24), spacing=_spacing(rng),
                    levels=rng.randint(1, 2), iters=rng.randint(2, 4))
    sizes = [_dims(rng, _log_uniform(rng, 40.0 ** 3, 96.0 ** 3), 8, 32) for _ in range(rng.randint(2, 6))]
    return dict(kind=kind, levels=rng.randint(1, 2), iters=2, spacing=_spacing(rng), sizes=" ".join(sizes))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _generator(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + int(salt))
    return g


def _axes(count, step, offset):
    """Positions in mm of the points of a grid, shaped to broadcast as (z, y, x)."""
    out = []
    for d in range(3):
        a = (torch.arange(count[d], device="cuda", dtype=torch.float32) + offset) * step[d]
        shape = [1, 1, 1]
        shape[2 - d] = count[d]
        out.append(a.reshape(shape))
    return out


def _modes(rng, extent):
    """A smooth deformation: per component three sine modes, at most about 4 % of the extent."""
    return [[(rng.uniform(-0.5, 0.5), [rng.uniform(0.4, 1.6) * 2 * math.pi / e for e in extent],
              [rng.uniform(0, 2 * math.pi) for _ in range(3)]) for _ in range(3)] for _ in range(3)]


def _field(modes, ax, extent, scale):
    amp = scale * 0.04 * min(extent)
    out = []
    for comp in modes:
        f = 0.0
        for a, k, ph in comp:
            s = [torch.sin(ax[d] * k[d] + ph[d]) for d in range(3)]
            f = f + (a * amp) * (s[0] * s[1]) * s[2]
        out.append(f)
    return out


def _phantom(blobs, pos, extent):
    """Intensity at positions (x, y, z) in mm: a soft-edged body with organs in it."""
    c = [0.5 * e for e in extent]
    width = 0.02 * min(extent)
    r = torch.sqrt(sum(((pos[d] - c[d]) / (0.42 * extent[d])) ** 2 for d in range(3)))
    f = 0.6 * torch.sigmoid((1.0 - r) * (0.42 * min(extent) / width))
    for ctr, semi, level in blobs:
        r = torch.sqrt(sum(((pos[d] - ctr[d]) / semi[d]) ** 2 for d in range(3)))
        f = f + level * torch.sigmoid((1.0 - r) * (min(semi) / width))
    return f


def _pair(dims, spacing, seed):
    """R and T = R warped, each with its own noise, and the modes of the deformation between them."""
    rng = np.random.default_rng([int(seed), 17])
    extent = [dims[d] * spacing[d] for d in range(3)]
    blobs = []
    for i in range(10):
        semi = [rng.uniform(0.05, 0.2) * e for e in extent]
        ctr = [rng.uniform(0.25, 0.75) * e for e in extent]
        blobs.append((ctr, semi, rng.uniform(0.05, 0.3) * (1 if i & 1 else -1)))
    modes = _modes(rng, extent)
    ax = _axes(dims, spacing, 0.5)
    full = [a.expand(dims[2], dims[1], dims[0]) for a in ax]
    shift = _field(modes, ax, extent, 1.0)
    g = _generator(seed)
    out = []
    for pos in (full, [full[d] + shift[d] for d in range(3)]):
        img = _phantom(blobs, pos, extent)
        img = img + 0.012 * torch.randn(img.shape, generator=g, device="cuda")
        out.append(img.clamp_(0.0, 1.0).contiguous())
    return out[0], out[1], modes


def _displacement(nodes, dims, spacing, modes, seed):
    """A displacement on the way to the solution: part of the true one, slightly uneven."""
    extent = [dims[d] * spacing[d] for d in range(3)]
    step = [extent[d] / (nodes[d] - 1) for d in range(3)]
    f = _field(modes, _axes(nodes, step, 0.0), extent, -0.7)
    u = torch.stack([c.expand(nodes[2], nodes[1], nodes[0]) for c in f])
    noise = torch.randn(u.shape, generator=_generator(seed, 1), device="cuda")
    return (u + 0.02 * min(spacing) * noise).contiguous()


def _nodes(case):
    per = 2 if case["nodes"] == "half" else 4
    return [max(3, m // per + 1) for m in _sizes(case["dims"])]


def _handle(case, levels=1):
    kw = {}
    if case.get("nodes") == "quarter":
        kw["node_dims"] = [_nodes(case)]
    return reg.Registration(reg.make_config(levels=levels, tau=TAU, alpha=ALPHA, mem=MEM,
                                            image_dtype=case.get("dtype", "f32"), **kw))


def prepare(case, seed):
    kind, h = case["kind"], _mm(case) if "spacing" in case else None
    state = dict(case=case, kind=kind, spacing=h)
    if kind in ("eval", "autograd"):
        dims = _sizes(case["dims"])
        R, T, modes = _pair(dims, h, seed)
        state["reg"] = _handle(case).set_images(R, T, h)
        state["u"] = _displacement(_nodes(case), dims, h, modes, seed)
        if kind == "autograd":
            state["u"].requires_grad_(True)
    elif kind == "images":
        # the handle has held another frame of the same geometry before
        R0, T0, _ = _pair(_sizes(case["dims"]), h, seed + 7919)
        state["reg"] = _handle(case, case["levels"]).set_images(R0, T0, h)
        state["R"], state["T"], _ = _pair(_sizes(case["dims"]), h, seed)
    elif kind == "direction":
        R, T, _ = _pair([16, 16, 16], [1.0, 1.0, 1.0], seed)
        cfg = reg.make_config(levels=1, tau=TAU, alpha=ALPHA, mem=max(MEM, case["count"]))
        state["reg"] = reg.Registration(cfg).set_images(R, T, [1.0, 1.0, 1.0])
        state["S"], state["Y"], state["g"] = _lbfgs_pairs(case, seed)
    elif kind == "register":
        dims = _sizes(case["dims"])
        state["R"], state["T"], modes = _pair(dims, h, seed)
        coarse = _level_dims(dims, case["levels"] - 1)
        state["u"] = _displacement([m // 2 + 1 for m in coarse], dims, h, modes, seed)
    else:
        cfg = reg.make_config(levels=case["levels"], tau=TAU, alpha=ALPHA, mem=MEM, max_iter=case["iters"],
                              fixed_iters=True)
        state["regs"] = []
        for i, d in enumerate(case["sizes"].split()):
            R, T, _ = _pair(_sizes(d), h, 1000 * seed + i)
            state["regs"].append(reg.Registration(cfg).set_images(R, T, h))
    return state


def _lbfgs_pairs(case, seed):
    """Steps, gradient differences (positive curvature) and a gradient of an elastic-like problem."""
    n = 3 * _voxels(_sizes(case["nodes"]))
    g = _generator(seed, 2)
    c = case["count"]
    stiff = 0.5 + 2.5 * torch.rand(n, generator=g, device="cuda")
    S = torch.randn((c, n), generator=g, device="cuda")
    Y = S * stiff + 0.05 * torch.randn((c, n), generator=g, device="cuda")
    return S, Y, torch.randn(n, generator=g, device="cuda")


def _made_levels(case):
    """The pyramid levels that the call computes (level 0 is the input)."""
    return range(1, case["levels"])


def _scalars(J, D, S):
    return np.array([J, D, S], dtype=np.float32)


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "eval":
        J, D, S, grad = state["reg"].eval(state["u"])
        return {"JDS": _scalars(J, D, S), "grad": grad}
    if kind == "autograd":
        u = state["u"]
        u.grad = None
        J = reg.RegObjective.apply(u, state["reg"])
        J.backward()
        return {"J": J.detach().float(), "grad": u.grad}
    if kind == "images":
        r = state["reg"].set_images(state["R"], state["T"], state["spacing"])
        return {"%s%d" % (w, lv): r.level_image(lv, w) for lv in _made_levels(case) for w in "RT"}
    if kind == "direction":
        return state["reg"].lbfgs_direction(state["S"], state["Y"], state["g"])
    if kind == "register":
        u, st = reg.register(state["R"], state["T"], state["spacing"], u_init=state["u"], levels=case["levels"],
                             tau=TAU, alpha=ALPHA, mem=MEM, max_iter=case["iters"], fixed_iters=True)
        return {"u": u, "JDS": _scalars(st["J_final"], st["D_final"], st["S_final"]), "iters": st["iters"],
                "evals": st["evals"]}
    out = reg.register_batch(state["regs"])
    return [{"u": u, "JDS": _scalars(st["J_final"], st["D_final"], st["S_final"]), "iters": st["iters"],
             "evals": st["evals"]} for u, st in out]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
EVAL_FLOPS = 200           # per voxel: P, interpolation with gradient, NGF and its adjoint, P^T


def _voxels(d):
    return d[0] * d[1] * d[2]


def _level_dims(dims, level):
    for _ in range(level):
        dims = [(m + 1) // 2 for m in dims]
    return dims


def _eval_work(dims, nodes, image_bytes=4):
    """Read R, T and u, write the gradient."""
    nv, nn = _voxels(dims), _voxels(nodes)
    return 2 * image_bytes * nv + 24 * nn, EVAL_FLOPS * nv


def _solve_work(dims, levels, iters):
    """Images in, pyramid out, one evaluation and one pass over u, g and the pairs per iteration, u out."""
    b, f = 8 * _voxels(dims), 0
    for lv in range(levels):
        d = _level_dims(dims, lv)
        n = [m // 2 + 1 for m in d]
        eb, ef = _eval_work(d, n)
        vectors = sum(4 + 2 * min(i, MEM) for i in range(iters)) * 12 * _voxels(n)
        b += (iters + 1) * eb + vectors
        f += (iters + 1) * ef + vectors // 2
    return b + 12 * _voxels([m // 2 + 1 for m in dims]), f


def work(case):
    kind = case["kind"]
    if kind in ("eval", "autograd"):
        b, f = _eval_work(_sizes(case["dims"]), _nodes(case), 2 if case["dtype"] == "bf16" else 4)
    elif kind == "images":
        dims = _sizes(case["dims"])
        pyramid = sum(_voxels(_level_dims(dims, lv)) for lv in range(case["levels"]))
        b, f = 8 * _voxels(dims) + 8 * pyramid, 8 * pyramid
    elif kind == "direction":
        n = 3 * _voxels(_sizes(case["nodes"]))
        b, f = 4 * n * (2 * case["count"] + 2), n * (4 * case["count"] ** 2 + 8 * case["count"])
    elif kind == "register":
        b, f = _solve_work(_sizes(case["dims"]), case["levels"], case["iters"])
    else:
        parts = [_solve_work(_sizes(d), case["levels"], case["iters"]) for d in case["sizes"].split()]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _hat_matrix(m, n):
    """P along one axis: m voxel centres between n nodes on the same extent."""
    t = (torch.arange(m, dtype=torch.float64) + 0.5) * (n - 1) / m
    k = t.floor().clamp(0, n - 2).long()
    A = torch.zeros((m, n), dtype=torch.float64)
    i = torch.arange(m)
    A[i, k] = 1.0 - (t - k)
    A[i, k + 1] = t - k
    return A.cuda()


def _along(A, x):
    """Apply the matrices (x, y, z order) along the axes of a (z, y, x) volume."""
    x = torch.matmul(x, A[0].T)
    x = torch.matmul(A[1], x)
    return torch.tensordot(A[2], x, dims=1)


def _shifted(x, axis, step):
    """The interior neighbours x[i + step] along an axis, same shape, zero beyond the ends."""
    y = torch.zeros_like(x)
    n = x.shape[axis]
    if step > 0:
        y.narrow(axis, 0, n - 1).copy_(x.narrow(axis, 1, n - 1))
    else:
        y.narrow(axis, 1, n - 1).copy_(x.narrow(axis, 0, n - 1))
    return y


def _interpolate(T, pos):
    """Trilinear value of T and its interpolant's gradient (per voxel) at voxel coordinates, zero outside."""
    m = [T.shape[2], T.shape[1], T.shape[0]]
    cell = [p.floor() for p in pos]
    f = [p - c for p, c in zip(pos, cell)]
    flat, corner = T.reshape(-1), []
    for j in range(8):
        idx = [cell[d].long() + ((j >> d) & 1) for d in range(3)]
        inside = torch.ones_like(idx[0], dtype=torch.bool)
        for d in range(3):
            inside &= (idx[d] >= 0) & (idx[d] < m[d])
            idx[d].clamp_(0, m[d] - 1)
        corner.append(torch.where(inside, flat[(idx[2] * m[1] + idx[1]) * m[0] + idx[0]], 0.0))
    d00, d10, d01, d11 = (corner[j + 1] - corner[j] for j in (0, 2, 4, 6))
    a00, a10, a01, a11 = corner[0] + f[0] * d00, corner[2] + f[0] * d10, corner[4] + f[0] * d01, corner[6] + f[0] * d11
    e0, e1 = a10 - a00, a11 - a01
    b0, b1 = a00 + f[1] * e0, a01 + f[1] * e1
    gx0, gx1 = d00 + f[1] * (d10 - d00), d01 + f[1] * (d11 - d01)
    return b0 + f[2] * (b1 - b0), [gx0 + f[2] * (gx1 - gx0), e0 + f[2] * (e1 - e0), b1 - b0]


def _objective64(R, T, spacing, u, tau, alpha):
    """J, D, S and the gradient of the objective (Eq. 1 and 2) in 64 bits."""
    R, T, u = R.double(), T.double(), u.double()
    m, n = [R.shape[2], R.shape[1], R.shape[0]], [u.shape[3], u.shape[2], u.shape[1]]
    h = [float(s) for s in spacing]
    A = [_hat_matrix(m[d], n[d]) for d in range(3)]
    pos = []
    for d in range(3):
        i = torch.arange(m[d], device="cuda", dtype=torch.float64)
        shape = [1, 1, 1]
        shape[2 - d] = m[d]
        pos.append(_along(A, u[d]) / h[d] + i.reshape(shape))
    W, dT = _interpolate(T, pos)
    del pos
    inner = torch.zeros_like(R)
    inner[1:-1, 1:-1, 1:-1] = 1.0
    a = [(_shifted(W, 2 - d, 1) - _shifted(W, 2 - d, -1)) * (inner / (2 * h[d])) for d in range(3)]
    b = [(_shifted(R, 2 - d, 1) - _shifted(R, 2 - d, -1)) * (inner / (2 * h[d])) for d in range(3)]
    na2 = sum(x * x for x in a) + tau * tau
    nb2 = sum(x * x for x in b) + tau * tau
    dot = sum(x * y for x, y in zip(a, b)) + tau * tau
    hbar = h[0] * h[1] * h[2]
    D = 0.5 * hbar * float(((1.0 - dot * dot / (na2 * nb2)) * inner).sum())
    k1, k2 = -2.0 * dot / (na2 * nb2) * inner, 2.0 * dot * dot / (na2 * na2 * nb2) * inner
    g = torch.zeros_like(R)
    for d in range(3):
        v = k1 * b[d] + k2 * a[d]
        g += (_shifted(v, 2 - d, -1) - _shifted(v, 2 - d, 1)) / (2 * h[d])
    g *= 0.5 * hbar
    H = [m[d] * h[d] / (n[d] - 1) for d in range(3)]
    hy = H[0] * H[1] * H[2]
    mask = torch.zeros_like(u[0])
    mask[1:-1, 1:-1, 1:-1] = 1.0

    def laplace(x):
        return sum((_shifted(x, 2 - d, 1) - 2.0 * x + _shifted(x, 2 - d, -1)) / (H[d] * H[d]) for d in range(3))

    S, grad = 0.0, []
    for c in range(3):
        w = laplace(u[c]) * mask
        S += 0.5 * hy * float((w * w).sum())
        grad.append(_along([M.T for M in A], g * dT[c] / h[c]) + alpha * hy * laplace(w))
    return D + alpha * S, D, S, torch.stack(grad)


def _restrict64(x):
    for axis in range(3):
        if x.shape[axis] & 1:
            x = torch.cat([x, x.narrow(axis, x.shape[axis] - 1, 1)], axis)
    z, y, w = (s // 2 for s in x.shape)
    return x.reshape(z, 2, y, 2, w, 2).mean(dim=(1, 3, 5))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("eval", "autograd"):
        dims, h = _sizes(case["dims"]), _mm(case)
        R, T, modes = _pair(dims, h, seed)
        if case["dtype"] == "bf16":      # the images as that option stores them
            R, T = R.bfloat16().float(), T.bfloat16().float()
        u = _displacement(_nodes(case), dims, h, modes, seed)
        J, D, S, grad = _objective64(R, T, h, u, TAU, ALPHA)
        if kind == "autograd":
            return {"J": torch.tensor(J, dtype=torch.float64), "grad": grad}
        return {"JDS": np.array([J, D, S]), "grad": grad}
    if kind == "images":
        out, level = {}, [x.double() for x in _pair(_sizes(case["dims"]), _mm(case), seed)[:2]]
        for lv in _made_levels(case):
            level = [_restrict64(x) for x in level]
            out.update({"R%d" % lv: level[0], "T%d" % lv: level[1]})
        return out
    if kind == "direction":
        S, Y, g = (x.double() for x in _lbfgs_pairs(case, seed))
        q, coef = g.clone(), []
        for s, y in zip(reversed(list(S)), reversed(list(Y))):
            coef.append((s @ q) / (s @ y))
            q -= coef[-1] * y
        q *= (S[-1] @ Y[-1]) / (Y[-1] @ Y[-1])
        for s, y, a in zip(S, Y, reversed(coef)):
            q += s * (a - (y @ q) / (s @ y))
        return -q
    return None

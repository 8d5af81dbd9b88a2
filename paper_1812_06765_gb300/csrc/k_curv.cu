// Curvature regulariser (Sec. 2.1: penalises (Laplace y_c)^2, Fischer and
// Modersitzki) and the final assembly J = D + alpha S (Eq. 1).
//
//   w_c = mask_interior * L u_c          (7-point Laplacian, node spacing H)
//   S   = hbar_y / 2 sum_c sum_k w_c^2
//   grad_c J += alpha hbar_y L^T w_c     (the symmetric stencil gathered over
//                                         the zero-extended w)
// Both passes are node-parallel, all 3 components of a node in one thread (the
// first takes up to 4 node planes per thread).
#include "internal.h"
#include "ngf_math.cuh"

namespace {

// element at a 32-bit byte offset from a base that is the same for the whole
// grid: one address register instead of 64-bit arithmetic per load (a plane
// array of one component holds less than 2^32 bytes, as 3 hold < 2^31 elements)
__device__ __forceinline__ float ld_at(const float *base, unsigned byte)
{
    return __ldg(reinterpret_cast<const float *>(reinterpret_cast<const char *>(base) + byte));
}

// A block takes CURV_NODES consecutive nodes of a plane (no lane idles at the
// end of a row) on curv_planes() node planes.  The z neighbours move up through
// registers, the x and y ones come from L1 at 32-bit offsets (a border node's
// missing neighbour reads the node itself; its w is masked).  HAS_DIR: at
// u + t dir.  The NGF pass's CTAs hold the whole register file, so this kernel
// runs before them or in their tail, and its time counts: 129^3 nodes 28 ->
// 19.5 us, 371 -> 154 instructions a node (one plane of 32 x 8 nodes a block,
// 64-bit addresses).  Past 4 planes a thread the gain is gone: fewer blocks
// than a wave or two.
template <bool HAS_DIR>
__global__ void __launch_bounds__(CURV_NODES) k_curv_w(LevelGeom g, const float *__restrict__ ub,
                                                         const float *__restrict__ dir,
                                                         const double *__restrict__ t_dev, float *__restrict__ w,
                                                         double *__restrict__ partials, int planes)
{
    __shared__ double sm[8];
    const int n0 = g.n[0];
    const int i = blockIdx.x * CURV_NODES + threadIdx.x;
    const int z0 = blockIdx.y * planes, z1 = min(g.n[2], z0 + planes);
    const float t = HAS_DIR ? (float)__ldg(t_dev) : 0.f;
    KahanF acc;
    if (i < n0 * g.n[1]) {
        const int y = i / n0, x = i - y * n0;
        const bool inxy = x >= 1 && y >= 1 && x <= n0 - 2 && y <= g.n[1] - 2;
        const unsigned plane = 4u * n0 * g.n[1];
        unsigned o = 4u * i + plane * z0;
        unsigned xm = inxy ? o - 4u : o, xp = inxy ? o + 4u : o;
        unsigned ym = inxy ? o - 4u * n0 : o, yp = inxy ? o + 4u * n0 : o;
        // the trial value, as the accepted update forms it
        auto node = [&](int d, unsigned b) {
            const float v = ld_at(ub + d * g.nn, b);
            return HAS_DIR ? fmaf(t, ld_at(dir + d * g.nn, b), v) : v;
        };
        float m[3], c[3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            m[d] = node(d, z0 > 0 ? o - plane : o);
            c[d] = node(d, o);
        }
        for (int z = z0; z < z1; z++) {
            const bool top = z == g.n[2] - 1, in = inxy && z >= 1 && !top;
            const unsigned up = top ? o : o + plane;
            float sq = 0.f;
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const float p = node(d, up);
                float lap = fmaf(node(d, xp) - 2.f * c[d] + node(d, xm), g.iH2[0], 0.f);
                lap = fmaf(node(d, yp) - 2.f * c[d] + node(d, ym), g.iH2[1], lap);
                lap = fmaf(p - 2.f * c[d] + m[d], g.iH2[2], lap);
                lap = in ? lap : 0.f;
                *reinterpret_cast<float *>(reinterpret_cast<char *>(w + d * g.nn) + o) = lap;
                sq = fmaf(lap, lap, sq);
                m[d] = c[d];
                c[d] = p;
            }
            acc.add(sq);
            o += plane;
            xm += plane;
            xp += plane;
            ym += plane;
            yp += plane;
        }
    }
    const double s = block_sum_to_f64(acc.s, sm);
    if (linear_tid() == 0)
        partials[linear_bid()] = s;
}

__global__ void __launch_bounds__(256) k_curv_grad(LevelGeom g, const float *__restrict__ w, float alpha_hy,
                                                   float *__restrict__ grad)
{
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    int y = blockIdx.y * blockDim.y + threadIdx.y;
    int z = blockIdx.z;
    if (x >= g.n[0] || y >= g.n[1])
        return;
    size_t k = x + (size_t)g.n[0] * (y + (size_t)g.n[1] * z);
    size_t st[3] = {1, (size_t)g.n[0], (size_t)g.n[0] * g.n[1]};
    int j[3] = {x, y, z};
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float *wc = w + c * g.nn;
        float w0 = __ldg(wc + k);
        float s = 0.f;
#pragma unroll
        for (int e = 0; e < 3; e++) {
            float lo = j[e] > 0 ? __ldg(wc + k - st[e]) : 0.f;
            float hi = j[e] < g.n[e] - 1 ? __ldg(wc + k + st[e]) : 0.f;
            s = fmaf(lo + hi - 2.f * w0, g.iH2[e], s);
        }
        grad[c * g.nn + k] = fmaf(alpha_hy, s, grad[c * g.nn + k]);
    }
}

__global__ void __launch_bounds__(512) k_finalize(const double *__restrict__ pD, int nD,
                                                  const double *__restrict__ pS, int nS, double hbar_half,
                                                  double alpha, double hy_half, double *__restrict__ scal)
{
    finalize_body(pD, nD, pS, nS, hbar_half, alpha, hy_half, scal);
}

}  // namespace

bool is_curv_w_kernel(const void *f)
{
    return f == reinterpret_cast<const void *>(k_curv_w<true>) || f == reinterpret_cast<const void *>(k_curv_w<false>);
}


cudaError_t launch_eval(reg_ctx *c, int level, const float *ub, const float *dir, const double *t_dev, float *grad,
                        double *scal_out, int ctl_phase, cudaStream_t s)
{
    const Level &L = c->L[level];
    LevelGeom g = L.geom();
    int nD = 0;
    cudaError_t e;
    const bool fused = use_fused(c, level), general = use_general(c, level);
    const bool curv_in_pass = fused && fused_curv_in_pass(c, level);
    // The curvature Laplacian (node pass, HBM-light) runs on the side stream
    // beside the NGF pass (issue-bound, two CTAs per SM that hold all its registers), in the tail of its last
    // wave: fork before, join before the gradient assembly.  Captured, the two
    // become parallel graph branches.  With the batched form's arithmetic the
    // fused pass forms it itself, with one S partial per tile.
    e = cudaSuccess;
    if (!curv_in_pass) {
        e = cudaEventRecord(c->ev_fork, s);
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(c->side, c->ev_fork, 0);
        if (e != cudaSuccess)
            return e;
    }
    if (c->time_ngf)
        e = cudaEventRecord(c->kev[0], s);
    if (e == cudaSuccess) {
        if (fused)
            e = launch_ngf_fused(c, level, ub, dir, t_dev, grad, c->es.partials, &nD, s);
        else if (general)
            e = launch_ngf_general(c, level, ub, dir, t_dev, &nD, s);
        else
            e = launch_ngf_multipass(c, level, ub, dir, t_dev, grad, c->es.partials, &nD, s);
    }
    if (e == cudaSuccess && c->time_ngf)
        e = cudaEventRecord(c->kev[1], s);
    if (e != cudaSuccess)
        return e;
    dim3 blk(32, 8, 1);
    dim3 gn((L.n[0] + 31) / 32, (L.n[1] + 7) / 8, L.n[2]);
    const int planes = curv_planes(L.n);
    const dim3 gw((L.n[0] * L.n[1] + CURV_NODES - 1) / CURV_NODES, (L.n[2] + planes - 1) / planes, 1);
    double *pS = c->es.partials + nD;
    if (!curv_in_pass) {
        dir ? k_curv_w<true><<<gw, CURV_NODES, 0, c->side>>>(g, ub, dir, t_dev, c->es.w, pS, planes)
            : k_curv_w<false><<<gw, CURV_NODES, 0, c->side>>>(g, ub, dir, t_dev, c->es.w, pS, planes);
        c->launches += 1;
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaEventRecord(c->ev_join, c->side);
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(s, c->ev_join, 0);
    }
    if (e != cudaSuccess)
        return e;
    double hy = L.H[0] * L.H[1] * L.H[2];
    int nS = curv_in_pass ? nD : (int)(gw.x * gw.y * gw.z);
    // grad = (tile partials of P^T r) + alpha hbar_y L^T w, and J, D, S (+ control).  The
    // final reduction reads only the block partials of the kernels before, not the
    // gradient.  On small grids block 0 of the gather runs it first (one launch); on
    // large ones it is a one-block kernel on the side stream beside the gather, since
    // the control code in the gather would cost the large grid occupancy.
    if (general && gather_blocks(L.n) < GATHER_SPLIT_BLOCKS)
        return launch_gather_general(c, level, c->es.w, (float)(c->cfg.alpha * hy), grad, true, nD, pS, nS, scal_out,
                                     ctl_phase, s);
    if (fused && gather_blocks(L.n) < GATHER_SPLIT_BLOCKS)
        return launch_gather_fin(c, level, c->es.w, (float)(c->cfg.alpha * hy), grad, nD, pS, nS, scal_out,
                                 ctl_phase, s);
    if (fused || general) {
        const double hbar = L.h[0] * L.h[1] * L.h[2];
        e = cudaEventRecord(c->ev_fork, s);
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(c->side, c->ev_fork, 0);
        if (e == cudaSuccess) {
            if (ctl_phase >= 0) {
                e = launch_finalize_ctl(c, c->es.partials, nD, pS, nS, 0.5 * hbar, c->cfg.alpha, 0.5 * hy, scal_out,
                                        ctl_phase, c->side);
            } else {
                k_finalize<<<1, 512, 0, c->side>>>(c->es.partials, nD, pS, nS, 0.5 * hbar, c->cfg.alpha, 0.5 * hy,
                                                    scal_out);
                e = cudaGetLastError();
            }
            c->launches += 1;
        }
        if (e == cudaSuccess && general)
            e = launch_gather_general(c, level, c->es.w, (float)(c->cfg.alpha * hy), grad, false, 0, nullptr, 0,
                                      nullptr, -1, s);
        else if (e == cudaSuccess)
            e = launch_gather_grad(c, level, c->es.w, (float)(c->cfg.alpha * hy), grad, s);
        if (e == cudaSuccess)
            e = cudaEventRecord(c->ev_join, c->side);
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(s, c->ev_join, 0);
        return e;
    }
    // multi-pass: grad += alpha hbar_y L^T w, then the final reduction
    k_curv_grad<<<gn, blk, 0, s>>>(g, c->es.w, (float)(c->cfg.alpha * hy), grad);
    double hbar = L.h[0] * L.h[1] * L.h[2];
    c->launches += 2;
    if (ctl_phase >= 0)   // the reduction block also takes the line-search decision
        return launch_finalize_ctl(c, c->es.partials, nD, pS, nS, 0.5 * hbar, c->cfg.alpha, 0.5 * hy, scal_out,
                                   ctl_phase, s);
    k_finalize<<<1, 512, 0, s>>>(c->es.partials, nD, pS, nS, 0.5 * hbar, c->cfg.alpha, 0.5 * hy, scal_out);
    return cudaGetLastError();
}

// Partial-sum slots one evaluation at this level needs (fused or multi-pass).
int eval_partials_needed(const Level &L)
{
    long long vox_blocks = (long long)((L.m[0] + 31) / 32) * ((L.m[1] + 7) / 8) * L.m[2];
    long long node_blocks = (long long)((L.n[0] + 31) / 32) * ((L.n[1] + 7) / 8) * L.n[2];
    return (int)(vox_blocks + node_blocks + 1024);
}

// Explicit-buffer launch of the final reduction, for callers that own every
// buffer (the allocation-free entry point).

cudaError_t launch_finalize_raw(const double *pD, int nD, const double *pS, int nS, double hbar_half, double alpha,
                                double hy_half, double *scal, cudaStream_t s)
{
    k_finalize<<<1, 512, 0, s>>>(pD, nD, pS, nS, hbar_half, alpha, hy_half, scal);
    return cudaGetLastError();
}

// Fused objective pass for grids of any ratio of at least 2 voxels per node
// interval in every dimension (odd image sizes, the quarter-resolution grids
// of Sec. 3.2, explicit node counts): the computation of the ratio-2 pass
// (k_ngf_fused.cu) with P and P^T from the per-dimension tables.
//
// It shares the ratio-2 pass's tile (16 x 16 threads, two adjacent voxel
// columns each, 28 x 12 output columns and a 2-voxel halo, a march along z),
// its packed arithmetic, its template with a zero border and R's normalized
// gradient field.  What differs:
//   P      the weights of a column and the nodes it lies between come from the
//          tables; the pair's columns lie in the same node interval or in
//          adjacent ones, so one 3 x 2 x 2 block of nodes serves both.  A plane
//          takes its weight from the table along z, and the block's node
//          planes advance when the plane's interval does (at most every other
//          plane at 2 voxels per interval).
//   P^T    r is first summed along z, in registers, into the two node planes of
//          the current interval.  When the interval is left its lower plane
//          is complete: the tile's columns of it go to shared memory, are
//          summed along x into node columns in the next step and along y
//          into the tile's partial in the step after.  So the x and y sums,
//          whose windows vary from node to node, run once per node plane
//          instead of once per voxel plane.
//
// What bounds it: as the ratio-2 pass, issue, latency and L1 together (181 x
// 217 x 181: 114 M warp instructions, issue active 0.54, L1 67 %, DRAM 11 %,
// 187 us).  The four kernels of the multi-pass form (k_ngf_multipass.cu) it
// replaces moved about 100 bytes per voxel through HBM and gathered P^T with
// scalar loads.  A whole evaluation, multi-pass -> this pass: 181 x 217 x 181
// with 91 x 109 x 91 nodes 415 -> 257 us, 256 x 256 x 112 with 65 x 65 x 29
// nodes 498 -> 233 us (equal z segments instead of the uneven split, and the
// x and y sums with run-time windows: 282 and 241 us); with the curvature and
// host side of the calls since, 237 and 220 us.
//
// Values that are not finite or out of range go as far as in the multi-pass
// kernels: a sample without a usable displacement is outside the image, a
// voxel reaches the nodes on which it has a weight, and the image's edges,
// which no interior difference reads, do not reach D.
#include "internal.h"
#include "lbfgs_control.cuh"

#include "fused_pass.cuh"

namespace {

// nodes that the 28 x 12 output columns of a tile reach at 2 or more voxels per interval
constexpr int GNX = 16, GNY = 8;
constexpr int GNE = 3 * GNX * GNY;                // partial entries per node plane (384)
// node tile of the 32 x 16 columns: 31 voxels span at most 16 intervals (17
// first nodes, and two nodes after the last), 15 at most 8
constexpr int GTX = 19, GTY = 10;
constexpr int GTP = 3 * GTY * GTX;                // floats of one node plane tile per array
constexpr int GSLOT_N = 3;                        // node planes: K and K + 1 in use while K + 2 is copied in
constexpr int GCOPY = (2 * GTP + NT - 1) / NT;
constexpr int GCOMB = (GTP + NT - 1) / NT;
constexpr int RROWS = OY;                         // rows of a completed node plane's columns
constexpr int TAPS = 5;                           // voxels of a node's two intervals, below 2.5 voxels per interval
static_assert(GNX == BX, "the x sums take one node column per thread of a row");

// shared layout (floats)
struct GSmem {
    static constexpr int T = 0;                          // T~ ring [4][PLANE]
    static constexpr int V = T + 4 * PLANE;              // v ring [4][3][PLANE]
    static constexpr int G = V + 12 * PLANE;             // grad T ring [GSLOTS][3][PLANE]
    static constexpr int RZ = G + GSLOTS * 3 * PLANE;    // r summed along z: [3][RROWS][CW]
    static constexpr int RX = RZ + 3 * RROWS * CW;       // summed along x too: [3][RROWS][GNX]
    static constexpr int N = RX + 3 * RROWS * GNX;       // node planes [GSLOT_N][2][GTP]
    static constexpr int WX = N + GSLOT_N * 2 * GTP;     // weight of node k0 + 1, per column [CW]
    static constexpr int WY = WX + CW;                   // per row [BY]
    static constexpr int WX0 = WY + BY;                  // weight of node k0 in P^T, per column [CW]
    static constexpr int WY0 = WX0 + CW;                 // per row [BY]
    static constexpr int KX = WY0 + BY;                  // k0 of the columns and rows (int)
    static constexpr int KY = KX + CW;
    static constexpr int FX = KY + BY;                   // first output column of each interval (int) [GNX + 2]
    static constexpr int FY = FX + GNX + 2;              // first output row [GNY + 2]
    static constexpr int BX0 = FY + GNY + 2;             // first output column with a weight on each node column (int) [GNX]
    static constexpr int BY0 = BX0 + GNX;                // first output row [GNY]
    static constexpr int TWX = BY0 + GNY;                // P^T weights of each node column [GNX][TAPS]
    static constexpr int TWY = TWX + GNX * TAPS;         // and node row [GNY][TAPS]
    static constexpr int FLOATS = TWY + GNY * TAPS;
    static constexpr size_t BYTES = sizeof(float) * FLOATS;
    static_assert(2 * (BYTES + 1024) <= 228 * 1024, "two CTAs of the general pass per SM");
    static_assert((V | G | RZ | RX | N | PLANE) % 2 == 0, "float2 rows need even offsets");
};

struct GenArgs {
    LevelGeom g;
    const void *T;          // zero-bordered template
    const float4 *Rn;       // R's normalized gradient field (row length rounded up to even)
    const float *ub, *dir;
    const double *t_dev;
    const float *pw0[3];    // P^T: weight of a voxel on its node k0, per dimension
    float tau;
    FusedSplit split;       // z segments
    int nseg;               // their count
    int ntx, nty;
    float *part;            // [tile column][n_z + 2 nseg][GNE]: node plane k of segment s at k + 2 s
    double *partials;       // D block partials, one per tile
};

// One output tile (launch-order id, see tile_seg_col).  FEW: no node has
// more than TAPS voxels in its two intervals along x or y (one that lies on the
// node before it counts too, with its weight of 0), and the x and y sums take
// exactly TAPS with weights from shared memory (zero where there are fewer): no
// loop counters or tests, about half the instructions of the general sums.
template <bool HAS_DIR, bool FEW>
__device__ __forceinline__ void general_tile(const GenArgs &a, int tile_id, float *sm)
{
    using SL = GSmem;
    const LevelGeom &g = a.g;
    const int tid = linear_tid(), tx = tid % BX, ty = tid / BX;
    const int sp = 2 * tx + CW * ty;
    const int ncols = a.ntx * a.nty;
    int seg, col, z0, tz;
    tile_seg_col(a.split, ncols, tile_id, seg, col);
    a.split.seg(seg, z0, tz);
    const int zend = z0 + tz;
    const int tile_y = col / a.ntx, tile_x = col - tile_y * a.ntx;
    const int x0 = tile_x * OX, y0 = tile_y * OY;
    const int xa = x0 - 2 + 2 * tx, y = y0 - 2 + ty;
    const int mx = g.m[0], my = g.m[1], mz = g.m[2];
    // the first column lies in the image (the second may lie one past an odd row:
    // R's field is zero there, so its v is, and the x sums leave it out)
    const bool col_in = xa >= 0 && xa < mx && y >= 0 && y < my;
    const float t = HAS_DIR ? (float)__ldg(a.t_dev) : 0.f;
    const float2 HX = bc2(0.5f * g.ih[0]), HY = bc2(0.5f * g.ih[1]), HZ = bc2(0.5f * g.ih[2]);
    const int MXP = mx + 4, MYP = my + 4;
    const size_t SXYP = (size_t)MXP * MYP;
    const unsigned CXM = (unsigned)mx + 2, CYM = (unsigned)my + 2, CZM = (unsigned)mz + 2;
    const int mxe = (mx + 1) & ~1;                // row length of R's field
    const size_t rn_plane = (size_t)mxe * my;
    const float4 *Rncol = a.Rn + (col_in ? xa + mxe * y : 0);
    const bool rowC = ty >= 2 && ty < BY - 2;
    const bool outxy = rowC && tx >= 1 && tx < BX - 1;
    const float2 MO = bc2(outxy ? 1.f : 0.f);     // psi is zero off the interior
    // T~ counts where an interior voxel's central differences read it: on the interior and beside it,
    // not on the image's edges or outside.  Bits 0, 1: of the pair's columns on the interior planes,
    // 2, 3: on the first and the last plane.
    // border coordinates of the pair's columns in x and y (4: outside).  T~ counts where an interior
    // voxel's central differences read it: on the interior and beside it, at most one border
    // coordinate with that of z; not on the image's edges or outside.
    auto cls = [](int i, int m) { return i < 0 || i >= m ? 4 : i == 0 || i == m - 1 ? 1 : 0; };
    const int c0 = cls(xa, mx) + cls(y, my), c1 = cls(xa + 1, mx) + cls(y, my);
    const int dyp = ty < BY - 1 ? CW : 0, dym = ty > 0 ? CW : 0;
    const int nz = g.n[2];
    const size_t node_plane = (size_t)g.n[0] * g.n[1];

    // tables of the tile's columns and rows (positions outside the image take the border's)
    int *kxs = reinterpret_cast<int *>(sm + SL::KX), *kys = reinterpret_cast<int *>(sm + SL::KY);
    int *fx = reinterpret_cast<int *>(sm + SL::FX), *fy = reinterpret_cast<int *>(sm + SL::FY);
    int *bx = reinterpret_cast<int *>(sm + SL::BX0), *by = reinterpret_cast<int *>(sm + SL::BY0);
    if (tid < CW) {
        const int i = min(max(x0 - 2 + tid, 0), mx - 1);
        kxs[tid] = __ldg(g.pk0[0] + i);
        sm[SL::WX + tid] = __ldg(g.pw1[0] + i);
        sm[SL::WX0 + tid] = __ldg(a.pw0[0] + i);
    } else if (tid >= 64 && tid < 64 + BY) {
        const int i = min(max(y0 - 2 + tid - 64, 0), my - 1);
        kys[tid - 64] = __ldg(g.pk0[1] + i);
        sm[SL::WY + tid - 64] = __ldg(g.pw1[1] + i);
        sm[SL::WY0 + tid - 64] = __ldg(a.pw0[1] + i);
    }
    __syncthreads();
    const int kx0 = kxs[0], ky0 = kys[0];                      // first node of the node tile
    const int ocx = min(OX, mx - x0), ocy = min(OY, my - y0);  // output columns and rows in the image
    const int kox = kxs[2], koy = kys[2];                      // first node of the output columns
    const int nxl = kxs[1 + ocx] - kox + 2, nyl = kys[1 + ocy] - koy + 2;   // nodes they reach
    // f[j + 1]: the first output column (row) in an interval >= j, for j = -1 .. GNX.  b[j]: that of the
    // interval before node j, less one that lies on the node before (weight 0: a value there that is
    // not finite must not reach node j)
    if (tid < GNX + 2) {
        int f = 2, b = 2;
        for (int i = 2; i < 2 + ocx; i++) {
            const int k = kxs[i] - kox - (tid - 1);
            f += k < 0;
            b += k < 0 || (k == 0 && sm[SL::WX + i] == 0.f);
        }
        fx[tid] = f;
        if (tid < GNX)
            bx[tid] = b;
    } else if (tid >= 64 && tid < 64 + GNY + 2) {
        int f = 2, b = 2;
        for (int i = 2; i < 2 + ocy; i++) {
            const int k = kys[i] - koy - (tid - 65);
            f += k < 0;
            b += k < 0 || (k == 0 && sm[SL::WY + i] == 0.f);
        }
        fy[tid - 64] = f;
        if (tid - 64 < GNY)
            by[tid - 64] = b;
    }
    // the pair's node intervals: the second column lies in the first's or the next one
    const int lkx = kxs[2 * tx] - kx0, lky = kys[ty] - ky0;
    const bool next = kxs[2 * tx + 1] != kxs[2 * tx];
    const float2 WXv = make_float2(sm[SL::WX + 2 * tx], sm[SL::WX + 2 * tx + 1]);
    const float2 WYv = bc2(sm[SL::WY + ty]);

    // cooperative copy of a node plane's tile
    int csrc[GCOPY];
#pragma unroll
    for (int q = 0; q < GCOPY; q++) {
        const int e = tid + q * NT, r = e >= GTP ? e - GTP : e;
        const int c = r / (GTY * GTX), r2 = r - c * (GTY * GTX);
        const int ly = r2 / GTX, lx = r2 - ly * GTX;
        const bool in = e < (HAS_DIR ? 2 : 1) * GTP && kx0 + lx < g.n[0] && ky0 + ly < g.n[1];
        csrc[q] = in ? (int)(c * g.nn) + kx0 + lx + g.n[0] * (ky0 + ly) : -1;
    }
    auto issue_plane = [&](int K) {
        float *dst = sm + SL::N + (K % GSLOT_N) * 2 * GTP;
        const bool kin = K < nz;
        const size_t kofs = kin ? node_plane * (size_t)K : 0;
#pragma unroll
        for (int q = 0; q < GCOPY; q++) {
            const int e = tid + q * NT;
            if (e < (HAS_DIR ? 2 : 1) * GTP) {
                const bool in = kin && csrc[q] >= 0;
                const float *base = e >= GTP ? a.dir : a.ub;
                cp_async4(dst + e, in ? base + kofs + csrc[q] : a.ub, in);
            }
        }
        cp_async_commit();
    };
    auto trial_plane = [&](int K) {   // u <- u + t dir in place, as the accepted update
        float *nu = sm + SL::N + (K % GSLOT_N) * 2 * GTP;
#pragma unroll
        for (int q = 0; q < GCOMB; q++) {
            const int e = tid + q * NT;
            if (e < GTP)
                nu[e] = fmaf(t, nu[e + GTP], nu[e]);
        }
    };
    // values of component c of a row of node plane K at the first and second node of either column
    auto node_row = [&](const float *p, float2 &a, float2 &b) {
        const float u0 = p[0], u1 = p[1], u2 = p[2];
        a = make_float2(u0, next ? u1 : u0);
        b = make_float2(u1, next ? u2 : u1);
    };
    auto zclamp = [&](int z) { return min(max(z, 0), mz - 1); };

    int Kcur = -1;                 // node interval of the plane issued last
    int pend = -1;                 // node plane copied in, its trial values still to form
    // Per column, of the interval: the in-plane interpolation of the node differences to the
    // value at the first node, on the lower and the upper node plane, and that value less its
    // whole voxels (rem) - the operations of sample_coord and grid_convert_point, in their order,
    // so that a sample next to a cell face falls into the same cell in either implementation
    float2 Bl[3], Dd[3], rem[3];
    int cb[2][3] = {};             // integer bases of the sample cells (with MAGI taken off; z: + the plane)
    bool ok0 = true, ok1 = true;
    float2 pc[8], fr[3];
    float4 bn0 = make_float4(0.f, 0.f, 0.f, 0.f), bn1 = bn0;
    KahanF2 psi_sum;
    int gs = 0;
    // r summed along z into the lower and upper node plane of the interval of phase C
    float2 lo[3], hi[3];
#pragma unroll
    for (int c = 0; c < 3; c++)
        lo[c] = hi[c] = make_float2(0.f, 0.f);
    // tables along z, a step ahead: of the plane phase A issues next and of phase C's
    int kq = __ldg(g.pk0[2] + zclamp(z0 - 2));
    float wq = __ldg(g.pw1[2] + zclamp(z0 - 2));
    int kc = __ldg(g.pk0[2] + z0);
    float wc = __ldg(g.pw1[2] + z0), wc0 = __ldg(a.pw0[2] + z0);
    int Kc = kc;                   // node interval of phase C's sums
    int kx_pend = -1, ky_pend = -1;   // node planes whose x sums, y sums are due

    // ---- A-issue of plane z1: P at the pair (the interval's part when it is entered), the
    // coordinates, and the loads of the corners, first used one step later
    auto a_issue = [&](int z1, bool first) {
        const int K = kq;
        const float2 WZ = bc2(wq);
        const int zn = zclamp(z1 + 1);
        kq = __ldg(g.pk0[2] + zn);
        wq = __ldg(g.pw1[2] + zn);
        if (K != Kcur) {   // uniform over the CTA
            Kcur = K;
            const float *nl = sm + SL::N + (K % GSLOT_N) * 2 * GTP + lky * GTX + lkx;
            const float *nh = sm + SL::N + ((K + 1) % GSLOT_N) * 2 * GTP + lky * GTX + lkx;
            float2 q0max = make_float2(0.f, 0.f), acc = q0max;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const int o = c * (GTY * GTX);
                float2 u0, d100, d010, d110, d001, d101, d011, d111;
                node_row(nl + o, u0, d100);
                node_row(nl + o + GTX, d010, d110);
                node_row(nh + o, d001, d101);
                node_row(nh + o + GTX, d011, d111);
                d100 = sub2(d100, u0);
                d010 = sub2(d010, u0);
                d110 = sub2(d110, u0);
                d001 = sub2(d001, u0);
                d101 = sub2(d101, u0);
                d011 = sub2(d011, u0);
                d111 = sub2(d111, u0);
                Bl[c] = lerp2(mul2(WXv, d100), lerp2(d010, d110, WXv), WYv);
                Dd[c] = lerp2(lerp2(d001, d101, WXv), lerp2(d011, d111, WXv), WYv);
                const float ih = g.ih[c];
                const float2 q0 = mul2(u0, bc2(ih));
                const float2 qi = make_float2(floorf(q0.x), floorf(q0.y));
                rem[c] = make_float2(fmaf(-qi.x, g.h[c], u0.x), fmaf(-qi.y, g.h[c], u0.y));   // |rem| <~ h
                q0max = make_float2(fmaxf(q0max.x, fabsf(q0.x)), fmaxf(q0max.y, fabsf(q0.y)));
                const int base = (c == 0 ? xa : c == 1 ? y : 0) + 2 - MAGI;
                cb[0][c] = (int)qi.x + base;
                cb[1][c] = (int)qi.y + base + (c == 0 ? 1 : 0);
                const float2 b = mul2(Bl[c], bc2(ih)), d = mul2(Dd[c], bc2(ih));
                acc = fma2(b, b, fma2(d, d, acc));
            }
            // the displacement of every plane between them is below 1e6 voxels and finite
            ok0 = q0max.x < 1.0e6f && acc.x < 1.0e12f;
            ok1 = q0max.y < 1.0e6f && acc.y < 1.0e12f;
            // a first node out of range: unusable on every plane of the interval
            if (!(q0max.x < 1.0e6f))
                Bl[0].x = Dd[0].x = NAN;
            if (!(q0max.y < 1.0e6f))
                Bl[0].y = Dd[0].y = NAN;
            if (!first) {   // plane K - 1's slot
                issue_plane(K + 2);
                pend = K + 2;
            }
        } else if (HAS_DIR && pend >= 0) {   // copied a step ago: an interval holds two planes or more
            trial_plane(pend);
            pend = -1;
        }
        int ix[2][3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float2 f = mul2(add2(rem[c], lerp2(Bl[c], Dd[c], WZ)), bc2(g.ih[c]));
            const float2 fm = __fadd2_rd(f, bc2(MAGF));
            fr[c] = sub2(f, sub2(fm, bc2(MAGF)));
            ix[0][c] = __float_as_int(fm.x);
            ix[1][c] = __float_as_int(fm.y);
        }
        // An interval whose ends are not both in range (never in a registration that converges):
        // sample_coord's test of the plane itself.  An unusable sample has the value and the
        // gradient 0: its corners are zeros, and its fractions, which may not be finite, 0 too.
        bool use0 = ok0, use1 = ok1;
        if (!(ok0 && ok1)) {
            use0 = use1 = true;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const float2 q = mul2(lerp2(Bl[c], Dd[c], WZ), bc2(g.ih[c]));
                use0 = use0 && fabsf(q.x) < 1.0e6f;   // false for NaN
                use1 = use1 && fabsf(q.y) < 1.0e6f;
            }
#pragma unroll
            for (int c = 0; c < 3; c++)
                fr[c] = make_float2(use0 ? fr[c].x : 0.f, use1 ? fr[c].y : 0.f);
        }
#pragma unroll
        for (int k = 0; k < 2; k++) {
            float v[8];
            corners_padded(static_cast<const TemplateElem<float>::type *>(a.T), ix[k][0] + cb[k][0],
                           ix[k][1] + cb[k][1], ix[k][2] + cb[k][2] + z1, k ? use1 : use0, CXM, CYM, CZM, MXP, MYP, SXYP,
                           v);
#pragma unroll
            for (int j = 0; j < 8; j++) {
                if (k)
                    pc[j].y = v[j];
                else
                    pc[j].x = v[j];
            }
        }
    };

    // ---- sums along x of the columns at src into node columns at dst, one node column
    // per thread of an output row: the columns of interval j - 1 with the weight of
    // their upper node, those of interval j with that of their lower one
    auto x_sums = [&](const float *src, float *dst) {
        if (FEW && rowC) {   // node columns past nxl have zero weights
            const int e0 = min(fx[tx], CW - TAPS);
            const float *w = sm + SL::TWX + tx * TAPS, *r = src + (ty - 2) * CW + e0;
            float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
            for (int i = 0; i < TAPS; i++)
                if (w[i] != 0.f) {   // predicated: a value that is not finite reaches no node without a weight on it
                    s0 = fmaf(w[i], r[i], s0);
                    s1 = fmaf(w[i], r[RROWS * CW + i], s1);
                    s2 = fmaf(w[i], r[2 * RROWS * CW + i], s2);
                }
            float *d = dst + (ty - 2) * GNX + tx;
            d[0] = s0;
            d[RROWS * GNX] = s1;
            d[2 * RROWS * GNX] = s2;
        } else if (!FEW && rowC && tx < nxl) {
            const int e0 = bx[tx], e1 = fx[tx + 1], e2 = fx[tx + 2];
            const float *r = src + (ty - 2) * CW;
            float s0 = 0.f, s1 = 0.f, s2 = 0.f;
            for (int i = e0; i < e2; i++) {
                const float w = sm[(i < e1 ? SL::WX : SL::WX0) + i];
                s0 = fmaf(w, r[i], s0);
                s1 = fmaf(w, r[RROWS * CW + i], s1);
                s2 = fmaf(w, r[2 * RROWS * CW + i], s2);
            }
            float *d = dst + (ty - 2) * GNX + tx;
            d[0] = s0;
            d[RROWS * GNX] = s1;
            d[2 * RROWS * GNX] = s2;
        }
    };
    // ---- sums along y into the tile's partial of node plane K
    float *part_tile = a.part + ((size_t)col * (nz + 2 * a.nseg) + 2 * seg) * GNE;
    auto y_sums = [&](const float *src, int K) {
#pragma unroll
        for (int q = 0; q < (GNE + NT - 1) / NT; q++) {
            const int e = tid + q * NT;
            const int c = e / (GNX * GNY), jy = (e / GNX) % GNY, jx = e % GNX;
            if (FEW && e < GNE && jy < nyl && jx < nxl) {
                const int e0 = min(fy[jy], 2 + RROWS - TAPS);
                const float *w = sm + SL::TWY + jy * TAPS, *r = src + c * (RROWS * GNX) + (e0 - 2) * GNX + jx;
                float s = 0.f;
#pragma unroll
                for (int i = 0; i < TAPS; i++)
                    if (w[i] != 0.f)
                        s = fmaf(w[i], r[i * GNX], s);
                part_tile[(size_t)K * GNE + e] = s;
            } else if (!FEW && e < GNE && jy < nyl && jx < nxl) {
                const int e0 = by[jy], e1 = fy[jy + 1], e2 = fy[jy + 2];
                const float *r = src + c * (RROWS * GNX) + jx;
                float s = 0.f;
                for (int i = e0; i < e2; i++) {
                    s = fmaf(sm[(i < e1 ? SL::WY : SL::WY0) + i], r[(i - 2) * GNX], s);
                }
                part_tile[(size_t)K * GNE + e] = s;
            }
        }
    };
    auto store_plane = [&](float *dst, const float2 r[3]) {
        if (rowC) {
            float *d = dst + (ty - 2) * CW + 2 * tx;
            sts2(d, r[0]);
            sts2(d + RROWS * CW, r[1]);
            sts2(d + 2 * RROWS * CW, r[2]);
        }
    };

    // ---- one step of the pipeline (FULL: every phase is active)
    auto step = [&](int s, auto full_t) {
        constexpr bool FULL = decltype(full_t)::value;
        const int zA = z0 - 2 + s;
        // ---- A-finish: T~ and the interpolant differences on plane zA
        if (FULL || zA <= zend + 1) {
            float2 val, gx, gy, gz;
            interp_pair(pc, fr, val, gx, gy, gz);
            // T~ where it does not count is 0: R's field is 0 off the interior, and so are psi and v, but
            // not beside a T~ that is not finite.  (Selecting psi and v instead: 181 x 217 x 181 4 us
            // and 256 x 256 x 112 on 65 x 65 x 29 nodes 3 us more an evaluation.)
            const int lim = zA >= 1 && zA <= mz - 2 ? 1 : zA == 0 || zA == mz - 1 ? 0 : -1;
            val = make_float2(c0 <= lim ? val.x : 0.f, c1 <= lim ? val.y : 0.f);
            sts2(sm + SL::T + (zA & 3) * PLANE + sp, val);
            float *gq = sm + SL::G + gs * 3 * PLANE + sp;
            sts2(gq, gx);
            sts2(gq + PLANE, gy);
            sts2(gq + 2 * PLANE, gz);
        }
        if (FULL || zA <= zend)
            a_issue(zA + 1, false);
        // ---- B: v on plane zA - 2, and R's field at the next one
        const int zB = zA - 2;
        if (FULL || (zB >= z0 - 1 && zB <= zend)) {
            const float *Tr = sm + SL::T + sp;
            float2 v[3];
            const float2 psi = ngf_pair_rn<true>(Tr + (zB & 3) * PLANE, Tr + ((zB + 1) & 3) * PLANE,
                                           Tr + ((zB - 1) & 3) * PLANE, dyp, dym, bn0, bn1, HX, HY, HZ, a.tau, v);
            if (FULL || (zB >= z0 && zB < zend))
                psi_sum.add(mul2(psi, MO));
            float *vq = sm + SL::V + (zB & 3) * 3 * PLANE + sp;
            sts2(vq, v[0]);
            sts2(vq + PLANE, v[1]);
            sts2(vq + 2 * PLANE, v[2]);
        }
        const int zn = zB + 1;
        const bool ld = col_in && (FULL || (zn >= z0 - 1 && zn <= zend && zn >= 0 && zn < mz));
        if (!FULL)
            bn0 = bn1 = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 *q = Rncol + rn_plane * (size_t)(FULL || ld ? zn : 0);
        ld_once4(bn0, q, ld);
        ld_once4(bn1, q + 1, ld);
        // ---- sums due of a completed node plane (a plane completes at most every other step)
        if (ky_pend >= 0) {
            y_sums(sm + SL::RX, ky_pend);
            ky_pend = -1;
        }
        if (kx_pend >= 0) {
            x_sums(sm + SL::RZ, sm + SL::RX);
            ky_pend = kx_pend;
            kx_pend = -1;
        }
        // ---- C: r on plane zA - 4, summed along z into the interval's node planes
        const int zC = zA - 4;
        if (FULL || (zC >= z0 && zC < zend)) {
            const float w = wc, w0 = wc0;
            const int K = kc;
            const int z2 = zclamp(zC + 1);
            kc = __ldg(g.pk0[2] + z2);
            wc = __ldg(g.pw1[2] + z2);
            wc0 = __ldg(a.pw0[2] + z2);
            if (K != Kc) {   // the interval's lower plane is complete (uniform over the CTA)
                store_plane(sm + SL::RZ, lo);
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    lo[c] = hi[c];
                    hi[c] = make_float2(0.f, 0.f);
                }
                kx_pend = Kc;
                Kc = K;
            }
            if (rowC) {   // uniform per warp
                const float *V0 = sm + SL::V + (zC & 3) * 3 * PLANE + sp;
                const float2 vx = lds2(V0);
                const float vl = __shfl_up_sync(0xffffffffu, vx.y, 1, BX);
                const float vr = __shfl_down_sync(0xffffffffu, vx.x, 1, BX);
                const float *Vz = sm + SL::V + 2 * PLANE + sp;
                const float2 gj = adjoint_pair(V0, Vz + ((zC - 1) & 3) * 3 * PLANE, Vz + ((zC + 1) & 3) * 3 * PLANE, vx,
                                               vl, vr, HX, HY, HZ);
                const float *gq = sm + SL::G + (gs == GSLOTS - 1 ? 0 : gs + 1) * 3 * PLANE + sp;
                const float2 gh = mul2(gj, bc2(w)), gl = mul2(gj, bc2(w0));
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const float2 dT = lds2(gq + c * PLANE);
                    lo[c] = fma2(gl, dT, lo[c]);
                    if (w != 0.f)   // uniform; a plane on a node plane has no weight on the next one
                        hi[c] = fma2(gh, dT, hi[c]);
                }
            }
        }
        gs = gs == GSLOTS - 1 ? 0 : gs + 1;
        cp_async_wait_all();
        __syncthreads();
    };

    // prologue: the node planes of the first interval and of the next, which plane z0 - 1
    // may already enter, then the loads of plane z0 - 2
#pragma unroll
    for (int k = 0; k < GSLOT_N; k++)
        issue_plane(kq + k);
    cp_async_wait_all();
    __syncthreads();
    if (HAS_DIR) {
#pragma unroll
        for (int k = 0; k < GSLOT_N; k++)
            trial_plane(kq + k);
        __syncthreads();
    }
    if (FEW && tid < (GNX + GNY) * TAPS) {
        const bool isx = tid < GNX * TAPS;
        const int e = isx ? tid : tid - GNX * TAPS, j = e / TAPS;
        const int *f = (isx ? fx : fy) + j;
        const int i = e - j * TAPS + min(f[0], isx ? CW - TAPS : 2 + RROWS - TAPS);
        sm[(isx ? SL::TWX : SL::TWY) + e] =
            i < f[0] || i >= f[2] ? 0.f : sm[i < f[1] ? (isx ? SL::WX : SL::WY) + i : (isx ? SL::WX0 : SL::WY0) + i];
    }
    a_issue(z0 - 2, true);
    __syncthreads();

    // every phase is active from step 6 to step tz + 2; phase C ends at step tz + 5
    int s = 0;
    const int nsteps = tz + 6;
    for (; s < 6; s++)
        step(s, std::false_type{});
    for (; s <= tz + 2; s++)
        step(s, std::true_type{});
    for (; s < nsteps; s++)
        step(s, std::false_type{});
    // the segment's last two node planes (the grad T ring is free), after any sums still due
    static_assert(3 * RROWS * CW <= 3 * PLANE, "a completed plane fits a slot of the grad T ring");
    if (ky_pend >= 0) {
        y_sums(sm + SL::RX, ky_pend);
        ky_pend = -1;
    }
    if (kx_pend >= 0) {
        x_sums(sm + SL::RZ, sm + SL::RX);
        ky_pend = kx_pend;
    }
    store_plane(sm + SL::G, lo);
    store_plane(sm + SL::G + 3 * PLANE, hi);
    __syncthreads();
    if (ky_pend >= 0)
        y_sums(sm + SL::RX, ky_pend);
    x_sums(sm + SL::G, sm + SL::V);
    x_sums(sm + SL::G + 3 * PLANE, sm + SL::V + 3 * PLANE);
    __syncthreads();
    y_sums(sm + SL::V, Kc);
    y_sums(sm + SL::V + 3 * PLANE, Kc + 1);
    // a tile's total holds tens of thousands of terms (the multi-pass kernels round one of 256 to FP32)
    const float2 ps = psi_sum.s, pe = psi_sum.c;
    const double ssum = block_sum_to_f64(df_add(DFloat{ps.x, -pe.x}, DFloat{ps.y, -pe.y}),
                                         reinterpret_cast<DFloat *>(sm + SL::RZ));
    if (tid == 0)
        a.partials[tile_id] = ssum;
}

template <bool HAS_DIR, bool FEW>
__global__ void __launch_bounds__(NT, CTAS_PER_SM) k_ngf_general(GenArgs a)
{
    extern __shared__ float sm[];
    general_tile<HAS_DIR, FEW>(a, blockIdx.x, sm);
}

// segment (z order) of plane z
__device__ __forceinline__ int seg_of_plane(const FusedSplit &sp, int z)
{
    const int e1 = sp.n1 * sp.l1, e2 = e1 + sp.n2 * sp.l2;
    return z < e1 ? z / sp.l1 : z < e2 ? sp.n1 + (z - e1) / sp.l2 : sp.n1 + sp.n2;
}

// grad J at a node: the tile partials of every tile whose voxels the node
// reaches (usually one or two per dimension, more where a node interval is
// wider than a tile), tiles in x, y, z order, plus alpha hbar_y L^T w.  FIN:
// block 0 first reduces J, D and S (and takes the line-search decision).
struct GenFinArgs {
    const double *pD, *pS;
    int nD, nS;
    double hbar_half, alpha, hy_half;
    double *scal;
    int phase;
    LbfgsState *st;
    unsigned long long h_ls;
};

template <bool FIN>
__global__ void __launch_bounds__(GATHER_NODES) k_gather_general(GenArgs a, const float *__restrict__ w, float alpha_hy,
                                                                 float *__restrict__ grad, GenFinArgs f)
{
    if (FIN && blockIdx.x == 0 && blockIdx.y == 0) {
        finalize_body(f.pD, f.nD, f.pS, f.nS, f.hbar_half, f.alpha, f.hy_half, f.scal);
        if (f.phase >= 0) {
            __syncthreads();
            lb_control_body(f.phase, f.st, nullptr, nullptr, 0, f.scal, f.h_ls, 0ULL, 0ULL);
        }
    }
    const LevelGeom &g = a.g;
    const int n0 = g.n[0], n01 = g.n[0] * g.n[1];
    const int i = blockIdx.x * GATHER_NODES + threadIdx.x, kz = blockIdx.y;
    if (i >= n01)
        return;
    const int ky = i / n0, kx = i - ky * n0;
    const int fx = __ldg(g.tfirst[0] + kx), fy = __ldg(g.tfirst[1] + ky), fz = __ldg(g.tfirst[2] + kz);
    const int tx0 = fx / OX, tx1 = (fx + __ldg(g.tcnt[0] + kx) - 1) / OX;
    const int ty0 = fy / OY, ty1 = (fy + __ldg(g.tcnt[1] + ky) - 1) / OY;
    const int s0 = seg_of_plane(a.split, fz), s1 = seg_of_plane(a.split, fz + __ldg(g.tcnt[2] + kz) - 1);
    const size_t tile = (size_t)(g.n[2] + 2 * a.nseg) * GNE;
    float s[3] = {0.f, 0.f, 0.f};
    for (int sg = s0; sg <= s1; sg++)
        for (int ty = ty0; ty <= ty1; ty++) {
            const int jy = ky - __ldg(g.pk0[1] + ty * OY);
            for (int tx = tx0; tx <= tx1; tx++) {
                const int jx = kx - __ldg(g.pk0[0] + tx * OX);
                const float *p = a.part + (size_t)(tx + a.ntx * ty) * tile + (size_t)(kz + 2 * sg) * GNE + jy * GNX + jx;
                s[0] += __ldg(p);
                s[1] += __ldg(p + GNX * GNY);
                s[2] += __ldg(p + 2 * GNX * GNY);
            }
        }
    const float hh = 0.5f * g.hbar;
    const int k = i + n01 * kz;
    const int st[3] = {1, n0, n01};
    const int j[3] = {kx, ky, kz};
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float *wn = w + c * g.nn;
        const float w0 = __ldg(wn + k);
        float l = 0.f;
#pragma unroll
        for (int e = 0; e < 3; e++) {
            const float b = j[e] > 0 ? __ldg(wn + k - st[e]) : 0.f;
            const float t = j[e] < g.n[e] - 1 ? __ldg(wn + k + st[e]) : 0.f;
            l = fmaf(b + t - 2.f * w0, g.iH2[e], l);
        }
        grad[c * g.nn + k] = fmaf(alpha_hy, l, hh * g.ih[c] * s[c]);
    }
}

GenArgs general_args(const reg_ctx *c, int level, const float *ub, const float *dir, const double *t_dev)
{
    const Level &L = c->L[level];
    GenArgs a;
    a.g = L.geom();
    a.T = L.Tp;
    a.Rn = L.Rn;
    a.ub = ub;
    a.dir = dir;
    a.t_dev = t_dev;
    for (int d = 0; d < 3; d++)
        a.pw0[d] = L.pw0[d];
    a.tau = (float)c->cfg.tau;
    a.split = L.gen_split;
    a.nseg = L.gen_split.count();
    a.ntx = (L.m[0] + OX - 1) / OX;
    a.nty = (L.m[1] + OY - 1) / OY;
    a.part = c->es.part;
    a.partials = c->es.partials;
    return a;
}

}  // namespace

// At 2 or more voxels per node interval in every dimension a tile's columns
// reach at most GNX x GNY nodes and a node plane lasts two voxel planes or
// more.  Denser node grids keep the multi-pass kernels.
bool general_eligible(const Level &L)
{
    for (int d = 0; d < 3; d++)
        if (2 * (L.n[d] - 1) > L.m[d])
            return false;
    return true;
}

size_t general_part_floats(const Level &L)
{
    const size_t ncols = (size_t)((L.m[0] + OX - 1) / OX) * ((L.m[1] + OY - 1) / OY);
    return ncols * (size_t)(L.n[2] + 2 * L.gen_split.count()) * GNE;
}

cudaError_t launch_ngf_general(reg_ctx *c, int level, const float *ub, const float *dir, const double *t_dev,
                               int *n_partials, cudaStream_t s)
{
    static bool attr_set[64] = {};
    const int dev = c->device >= 0 && c->device < 64 ? c->device : 0;
    if (!attr_set[dev]) {
        cudaError_t e = set_fused_smem(k_ngf_general<true, true>, GSmem::BYTES);
        if (e == cudaSuccess)
            e = set_fused_smem(k_ngf_general<false, true>, GSmem::BYTES);
        if (e == cudaSuccess)
            e = set_fused_smem(k_ngf_general<true, false>, GSmem::BYTES);
        if (e == cudaSuccess)
            e = set_fused_smem(k_ngf_general<false, false>, GSmem::BYTES);
        if (e != cudaSuccess)
            return e;
        attr_set[dev] = true;
    }
    const GenArgs a = general_args(c, level, ub, dir, t_dev);
    *n_partials = a.ntx * a.nty * a.nseg;
    const dim3 blk(BX, BY, 1);
    const Level &L = c->L[level];
    if (L.reach[0] <= TAPS && L.reach[1] <= TAPS)
        dir ? k_ngf_general<true, true><<<*n_partials, blk, GSmem::BYTES, s>>>(a)
            : k_ngf_general<false, true><<<*n_partials, blk, GSmem::BYTES, s>>>(a);
    else
        dir ? k_ngf_general<true, false><<<*n_partials, blk, GSmem::BYTES, s>>>(a)
            : k_ngf_general<false, false><<<*n_partials, blk, GSmem::BYTES, s>>>(a);
    c->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_gather_general(reg_ctx *c, int level, const float *w, float alpha_hy, float *grad, bool fin, int nD,
                                  const double *pS, int nS, double *scal, int phase, cudaStream_t s)
{
    const Level &L = c->L[level];
    const GenArgs a = general_args(c, level, nullptr, nullptr, nullptr);
    GenFinArgs f = {};
    if (fin) {
        f.pD = c->es.partials;
        f.nD = nD;
        f.pS = pS;
        f.nS = nS;
        f.hbar_half = 0.5 * L.h[0] * L.h[1] * L.h[2];
        f.alpha = c->cfg.alpha;
        f.hy_half = 0.5 * L.H[0] * L.H[1] * L.H[2];
        f.scal = scal;
        f.phase = phase;
        f.st = c->lb.st;
        f.h_ls = phase >= 0 ? lbfgs_graph_handle_ls() : 0ULL;
        k_gather_general<true><<<gather_grid(L.n), GATHER_NODES, 0, s>>>(a, w, alpha_hy, grad, f);
    } else {
        k_gather_general<false><<<gather_grid(L.n), GATHER_NODES, 0, s>>>(a, w, alpha_hy, grad, f);
    }
    c->launches += 1;
    return cudaGetLastError();
}

// Pyramid generation and multilevel prolongation.
//
// Pyramid (Sec. 2.2 "Generating the multi-level pyramid"): each coarser level
// is the 2x2x2 mean of the finer one (an odd dimension replicates its last
// slab), spacing doubles.  The reference and template pyramids run on two
// streams.  Prolongation (Sec. 2.1, coarse-to-fine): nodal trilinear
// interpolation of the coarse displacement onto the finer nodes, with
// per-dimension (first node, weight) tables.
#include <type_traits>

#include "internal.h"

namespace {

// One thread per output voxel; a warp covers 32 consecutive x of one row, so
// the two input rows it reads are contiguous 64-float spans.  EVEN: even row
// length, both columns of a voxel in one 8-byte load.
template <bool EVEN>
__global__ void __launch_bounds__(256) k_restrict(const float *__restrict__ src, int mx, int my, int mz,
                                                  float *__restrict__ dst, int ox, int oy, int oz)
{
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    int y = blockIdx.y * blockDim.y + threadIdx.y;
    int z = blockIdx.z;
    if (x >= ox || y >= oy)
        return;
    int x0 = 2 * x, x1 = min(2 * x + 1, mx - 1);
    int y0 = 2 * y, y1 = min(2 * y + 1, my - 1);
    int z0 = 2 * z, z1 = min(2 * z + 1, mz - 1);
    size_t sy = (size_t)mx, sz = (size_t)mx * my;
    auto pair = [&](size_t row) {
        return EVEN ? __ldg(reinterpret_cast<const float2 *>(src + row) + x)
                    : make_float2(__ldg(src + row + x0), __ldg(src + row + x1));
    };
    const float2 a = pair(y0 * sy + z0 * sz), b = pair(y1 * sy + z0 * sz);
    const float2 c = pair(y0 * sy + z1 * sz), d = pair(y1 * sy + z1 * sz);
    const float s = a.x + a.y + b.x + b.y + c.x + c.y + d.x + d.y;
    dst[x + (size_t)ox * (y + (size_t)oy * z)] = 0.125f * s;
}

// One thread per fine node, all three components.
__global__ void k_prolong(const float *__restrict__ uc, int cx, int cy, int cz, float *__restrict__ uf, int fx,
                          int fy, int fz, const int *__restrict__ k0x, const int *__restrict__ k0y,
                          const int *__restrict__ k0z, const float *__restrict__ w1x,
                          const float *__restrict__ w1y, const float *__restrict__ w1z)
{
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    int y = blockIdx.y * blockDim.y + threadIdx.y;
    int z = blockIdx.z;
    if (x >= fx || y >= fy)
        return;
    int kx = k0x[x], ky = k0y[y], kz = k0z[z];
    float wx = w1x[x], wy = w1y[y], wz = w1z[z];
    size_t sy = (size_t)cx, sz = (size_t)cx * cy, ncs = (size_t)cx * cy * cz;
    size_t nfs = (size_t)fx * fy * fz;
    size_t b = kx + ky * sy + kz * sz;
    size_t o = x + (size_t)fx * (y + (size_t)fy * z);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float *u = uc + c * ncs;
        float a0 = lerpf(__ldg(u + b), __ldg(u + b + 1), wx);
        float a1 = lerpf(__ldg(u + b + sy), __ldg(u + b + sy + 1), wx);
        float a2 = lerpf(__ldg(u + b + sz), __ldg(u + b + sz + 1), wx);
        float a3 = lerpf(__ldg(u + b + sz + sy), __ldg(u + b + sz + sy + 1), wx);
        uf[c * nfs + o] = lerpf(lerpf(a0, a1, wy), lerpf(a2, a3, wy), wz);
    }
}

template <int V>
struct VecOf;
template <>
struct VecOf<1> {
    using type = unsigned;
};
template <>
struct VecOf<2> {
    using type = uint2;
};
template <>
struct VecOf<4> {
    using type = uint4;
};
// a 4-byte element of the padded array from the image's values at x and x + 1
template <typename TOUT>
__device__ __forceinline__ unsigned pad_elem(float v, float vn)
{
    if (std::is_same<TOUT, float>::value)
        return __float_as_uint(v);
    const __nv_bfloat162 b = __floats2bfloat162_rn(v, vn);
    return *reinterpret_cast<const unsigned *>(&b);
}

// Zero-bordered copy of a volume (dims m) into an array of dims m + 4 with the
// volume at offset 2 in every dimension, border included; BF16 elements hold
// (T[x], T[x + 1]).  A thread writes V consecutive elements of a row in one
// store: V = 4 and 2 for row lengths that are multiples of it, so that the
// stores are aligned and a pair of source columns is inside or outside as one.
// HBM-bound: 256 x 256 x 112 (58 MB) 27 -> 11 us against one element per thread; odd rows 27 -> 20 us.
template <typename TOUT, int V>
__global__ void __launch_bounds__(256) k_pad_template(const float *__restrict__ src, int mx, int my, int mz,
                                                      TOUT *__restrict__ dst)
{
    const int py = my + 4, pz = mz + 4, w = (mx + 4) / V;   // stores per row
    const int i = blockIdx.x * 256 + threadIdx.x;
    const int y = i / w, x = (i - y * w) * V;
    if (y >= py)
        return;
    const int sx = x - 2, sy = y - 2;
    for (int z = blockIdx.y; z < pz; z += gridDim.y) {
        const int sz = z - 2;
        const bool in = (unsigned)sy < (unsigned)my && (unsigned)sz < (unsigned)mz;
        const float *row = src + ((size_t)sz * my + sy) * mx;
        auto at = [&](int c) { return in && (unsigned)c < (unsigned)mx ? __ldg(row + c) : 0.f; };
        float v[V + 1];
        if (V == 1) {
            v[0] = at(sx);
        } else {
#pragma unroll
            for (int k = 0; k + 1 < V; k += 2) {
                const float2 p = in && (unsigned)(sx + k) < (unsigned)mx
                                     ? __ldg(reinterpret_cast<const float2 *>(row + sx + k))
                                     : make_float2(0.f, 0.f);
                v[k] = p.x;
                v[k + 1] = p.y;
            }
        }
        v[V] = std::is_same<TOUT, float>::value ? 0.f : at(sx + V);
        union {
            typename VecOf<V>::type q;
            unsigned e[V];
        } o;
#pragma unroll
        for (int k = 0; k < V; k++)
            o.e[k] = pad_elem<TOUT>(v[k], v[k + 1]);
        reinterpret_cast<typename VecOf<V>::type *>(dst)[((size_t)z * py + y) * w + x / V] = o.q;
    }
}

// R's values, with BF16 images rounded to BF16 (to nearest even)
template <bool BF16>
__device__ __forceinline__ float ld_ref(const float *p)
{
    const float v = __ldg(p);
    return BF16 ? __bfloat162float(__float2bfloat16_rn(v)) : v;
}
// columns x (even) and x + 1; EVEN: even row length, one aligned load
template <bool BF16, bool EVEN>
__device__ __forceinline__ float2 ld_ref_pair(const float *p)
{
    if (!EVEN)
        return make_float2(ld_ref<BF16>(p), ld_ref<BF16>(p + 1));
    const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
    return BF16 ? __bfloat1622float2(__float22bfloat162_rn(v)) : v;
}

// R's normalized gradient field for the fused pass (Eq. 2): R is fixed for the
// whole registration, so its part of every NGF term is formed once per level.
// Per voxel, with b the central-difference gradient of R (the differences
// times 1 / (2 h_c), as the pass forms grad T~): (b / ||b||_rho, rho / ||b||_rho),
// ||b||_rho = sqrt(|b|^2 + rho^2) with a correctly rounded square root and
// division; zero on voxels outside the interior, which Eq. 2's sum leaves out.
// Stored by pairs of columns (x even, x + 1: the two columns a thread of the
// pass holds), 8 floats per pair: bx, bx', by, by' | bz, bz', rho', rho'',
// so that every pair of lanes of the pass's packed arithmetic is one 8-byte
// half of a 16-byte load.  The row length is rounded up to even, so pair p of
// a row starts at float 8 p and the array has 4 floats per voxel of such rows,
// as a float4 per voxel.  A thread forms a pair on FIELD_PLANES planes, the z
// neighbours in registers, and stores it as two 16-byte halves.  HBM-bound
// (16 bytes written per voxel); a thread per voxel with 4-byte stores at
// stride 8 took 47 us at 256 x 256 x 112, and with four separate divisions
// (163 instructions a voxel) 42 us; now 29 us (86 instructions).
constexpr int FIELD_PLANES = 4;
// Voxels from which a thread of the field and of the padded copy takes several
// planes.  4 planes against 1, field + copy: 129 x 127 x 123 (2.0 M) 17.2
// against 19.8 us, 161 x 159 x 151 27.1 against 35.0, 255 x 257 x 113 53
// against 62, even rows within 2 us of each other; 97 x 95 x 91 and 96^3 (0.8 M)
// within 1 us, where too few blocks would be left on smaller volumes.
constexpr long long MARCH_FROM = 1 << 20;
// a / b, correctly rounded, from r = 1 / b correctly rounded: one residual
// correction of a r (Markstein's theorem, IBM J. Res. Dev. 34, 1990; b and r in
// the normal range, and |a| from 2^-102 up or 0: the residual of a smaller a
// underflows, and the last bit of a quotient may then differ).  Several
// quotients of one divisor share r.
__device__ __forceinline__ float quotient(float a, float b, float r)
{
    const float q = a * r;
    return fmaf(fmaf(-q, b, a), r, q);
}
template <bool BF16, bool EVEN>
__global__ void __launch_bounds__(256) k_ref_normal_field(const float *__restrict__ R, int mx, int my, int mz, float hx,
                                                          float hy, float hz, float rho, float4 *__restrict__ out, int planes)
{
    const int x = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z0 = blockIdx.z * planes, z1 = min(mz, z0 + planes);
    const int mxe = (mx + 1) & ~1;   // rows of an odd length carry one more column of zeros
    if (x >= mxe || y >= my)
        return;
    const size_t sy = (size_t)mx, sz = (size_t)mx * my;
    const float *p = R + x + sy * y + sz * z0;
    float4 *o = out + x + (size_t)mxe * (y + (size_t)my * z0);
    const bool iny = y >= 1 && y <= my - 2;
    const bool in0 = iny && x >= 1 && x <= mx - 2, in1 = iny && x + 1 <= mx - 2;
    // a pair holds an interior column: then both its columns and x - 1 or x + 2 are in the image
    const bool any = in0 || in1;
    const float2 zero = make_float2(0.f, 0.f);
    float2 below = any && z0 > 0 ? ld_ref_pair<BF16, EVEN>(p - sz) : zero, at = any ? ld_ref_pair<BF16, EVEN>(p) : zero;
    for (int z = z0; z < z1; z++, p += sz, o += (size_t)mxe * my) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        const float2 above = any && z < mz - 1 ? ld_ref_pair<BF16, EVEN>(p + sz) : zero;
        if (any && z >= 1 && z <= mz - 2) {
            const float2 up = ld_ref_pair<BF16, EVEN>(p + sy), dn = ld_ref_pair<BF16, EVEN>(p - sy);
            const float l = in0 ? ld_ref<BF16>(p - 1) : 0.f, r = in1 ? ld_ref<BF16>(p + 2) : 0.f;
            auto field = [&](float bx, float by, float bz, float &ox, float &oy, float &oz, float &orho) {
                const float nb = sqrtf(fmaf(bz, bz, fmaf(by, by, bx * bx)) + rho * rho);
                if (nb > 1e-30f && nb < 1e30f) {
                    const float r = __frcp_rn(nb);
                    ox = quotient(bx, nb, r);
                    oy = quotient(by, nb, r);
                    oz = quotient(bz, nb, r);
                    orho = quotient(rho, nb, r);
                } else {
                    ox = bx / nb;
                    oy = by / nb;
                    oz = bz / nb;
                    orho = rho / nb;
                }
            };
            if (in0)
                field((at.y - l) * hx, (up.x - dn.x) * hy, (above.x - below.x) * hz, a.x, a.z, b.x, b.z);
            if (in1)
                field((r - at.x) * hx, (up.y - dn.y) * hy, (above.y - below.y) * hz, a.y, a.w, b.y, b.w);
        }
        o[0] = a;
        o[1] = b;
        below = at;
        at = above;
    }
}

template <typename TOUT>
cudaError_t launch_pad(const float *src, const int m[3], TOUT *dst, cudaStream_t s)
{
    const int v = m[0] % 4 == 0 ? 4 : m[0] % 2 == 0 ? 2 : 1;
    const int stores = (m[0] + 4) / v * (m[1] + 4);   // per plane
    // large volumes: 4 planes per thread, so that its place in the plane is found once
    const int pz = (long long)m[0] * m[1] * m[2] >= MARCH_FROM ? (m[2] + 4 + 3) / 4 : m[2] + 4;
    const dim3 grd((stores + 255) / 256, pz < 65535 ? pz : 65535, 1);
    if (v == 4)
        k_pad_template<TOUT, 4><<<grd, 256, 0, s>>>(src, m[0], m[1], m[2], dst);
    else if (v == 2)
        k_pad_template<TOUT, 2><<<grd, 256, 0, s>>>(src, m[0], m[1], m[2], dst);
    else
        k_pad_template<TOUT, 1><<<grd, 256, 0, s>>>(src, m[0], m[1], m[2], dst);
    return cudaGetLastError();
}

template <bool BF16>
cudaError_t launch_field(const Level &L, double rho, cudaStream_t s)
{
    // the pass's difference factors: 0.5 * (float)(1 / h), as in grad T~
    const LevelGeom g = L.geom();
    const float hx = 0.5f * g.ih[0], hy = 0.5f * g.ih[1], hz = 0.5f * g.ih[2];
    const int pairs = (L.m[0] + 1) / 2;
    const dim3 blk(32, 8, 1);
    const int planes = L.nv >= MARCH_FROM ? FIELD_PLANES : 1;
    const dim3 grd((pairs + 31) / 32, (L.m[1] + 7) / 8, (L.m[2] + planes - 1) / planes);
    if (L.m[0] % 2 == 0)
        k_ref_normal_field<BF16, true><<<grd, blk, 0, s>>>(L.R, L.m[0], L.m[1], L.m[2], hx, hy, hz, (float)rho, L.Rn,
                                                         planes);
    else
        k_ref_normal_field<BF16, false><<<grd, blk, 0, s>>>(L.R, L.m[0], L.m[1], L.m[2], hx, hy, hz, (float)rho, L.Rn,
                                                         planes);
    return cudaGetLastError();
}

}  // namespace

long long padded_voxels(const int m[3]) { return (long long)(m[0] + 4) * (m[1] + 4) * (m[2] + 4); }

cudaError_t launch_pad_template(const float *src, const int m[3], float *dst, cudaStream_t s)
{
    return launch_pad(src, m, dst, s);
}

cudaError_t launch_pad_template(const float *src, const int m[3], __nv_bfloat162 *dst, cudaStream_t s)
{
    return launch_pad(src, m, dst, s);
}

cudaError_t launch_ref_normal_field(const Level &L, double rho, cudaStream_t s)
{
    return L.Tb ? launch_field<true>(L, rho, s) : launch_field<false>(L, rho, s);
}

cudaError_t launch_restrict(const float *src, const int m[3], float *dst, cudaStream_t s)
{
    int o[3] = {(m[0] + 1) / 2, (m[1] + 1) / 2, (m[2] + 1) / 2};
    dim3 blk(32, 8, 1);
    dim3 grd((o[0] + 31) / 32, (o[1] + 7) / 8, o[2]);
    if (m[0] % 2 == 0)
        k_restrict<true><<<grd, blk, 0, s>>>(src, m[0], m[1], m[2], dst, o[0], o[1], o[2]);
    else
        k_restrict<false><<<grd, blk, 0, s>>>(src, m[0], m[1], m[2], dst, o[0], o[1], o[2]);
    return cudaGetLastError();
}

cudaError_t launch_prolong(const Level &coarse, const Level &fine, const float *uc, float *uf, cudaStream_t s)
{
    dim3 blk(32, 8, 1);
    dim3 grd((fine.n[0] + 31) / 32, (fine.n[1] + 7) / 8, fine.n[2]);
    k_prolong<<<grd, blk, 0, s>>>(uc, coarse.n[0], coarse.n[1], coarse.n[2], uf, fine.n[0], fine.n[1], fine.n[2],
                                  fine.qk0[0], fine.qk0[1], fine.qk0[2], fine.qw1[0], fine.qw1[1], fine.qw1[2]);
    return cudaGetLastError();
}

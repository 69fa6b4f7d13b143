// sph_post.cu -- the post-processing phase (Sec. 4.3) as CUDA kernels: the fluid's
// volume-fraction field on a regular grid (surface reconstruction input), its iso-surface
// by marching tetrahedra, and a headless orthographic height map of the particles.
//
//  * field: phi(g) = sum_j (m / rho_j) W(|g - x_j|), the SPH interpolant (Sec. 3.2) of the
//    constant 1: about 1 inside the fluid, 0 outside.  The scene's particles are first
//    sorted into its cell grid (counting sort, then a rank by index inside each cell, so
//    the summation order and the result are reproducible).  On fine grids a warp then takes a
//    tile of nodes with the particles near it; on coarse ones a thread per node walks the
//    node's stencil of cells.
//  * mesh: each grid cube is split into the six tetrahedra around its diagonal from corner
//    0 to corner 7 (corner index = dx + 2 dy + 4 dz); per tetrahedron the corners above the
//    iso-level are cut off by one triangle (one or three corners above) or two (two
//    above), vertices interpolated linearly along the cut edges from the corner above to
//    the corner below (the same arithmetic in every cube sharing an edge), each triangle oriented
//    so its normal points from the corners above to those below, in cube order.
//  * height map: per particle, the pixels of its disk receive z + sqrt(R^2 - d^2) through
//    an atomic maximum on an order-preserving integer image of the float.
#include "sph.h"
#include "sph_sweep.cuh"

#include <algorithm>
#include <cmath>

namespace sph {

namespace {

constexpr int kPostBlock = 256;

// ------------------------------------------------------------------ field
__global__ void k_pf_hist(const float4 *__restrict__ pos, int64_t n, SceneDev sc, uint32_t *count,
                          uint32_t *key, uint32_t *slot)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 p = pos[i];
    const int32_t ix = cell_coord(p.x, sc.origin[0], sc.cell, sc.dims[0]);
    const int32_t iy = cell_coord(p.y, sc.origin[1], sc.cell, sc.dims[1]);
    const int32_t iz = cell_coord(p.z, sc.origin[2], sc.cell, sc.dims[2]);
    const uint32_t k = (uint32_t)ix + (uint32_t)sc.dims[0] * ((uint32_t)iy + (uint32_t)sc.dims[1] * (uint32_t)iz);
    key[i] = k;
    slot[i] = atomicAdd(&count[k], 1u);
}

// Place each particle in its cell's range (order inside a cell not yet fixed).
__global__ void k_pf_place(int64_t n, const uint32_t *__restrict__ key, const uint32_t *__restrict__ slot,
                           const uint32_t *__restrict__ start, uint32_t *cellidx)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    cellidx[start[key[i]] + slot[i]] = (uint32_t)i;
}

// Rank inside the cell by particle index (reproducible order) and write (x, m / rho), rho
// the particle's density of the last step (the rest density before the first step).
__global__ void k_pf_rank(const float4 *__restrict__ pos, const float4 *__restrict__ vel, int64_t n, float mass,
                          float rho0, const uint32_t *__restrict__ key, const uint32_t *__restrict__ start,
                          const uint32_t *__restrict__ cellidx, float4 *sorted)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const uint32_t i = cellidx[s];
    const uint32_t k = key[i];
    const uint32_t b = start[k], e = start[k + 1];
    uint32_t rank = 0;
    for (uint32_t t = b; t < e; ++t) rank += cellidx[t] < i ? 1u : 0u;
    const float4 p = pos[i];
    const float rho = vel[i].w;
    sorted[b + rank] = make_float4(p.x, p.y, p.z, mass / (rho > 0.0f ? rho : rho0));
}

__global__ void k_pf_field(const float4 *__restrict__ sorted, const uint32_t *__restrict__ start, SceneDev sc,
                           float ox, float oy, float oz, float spacing, int32_t nx, int32_t ny, int32_t nz,
                           float *__restrict__ out)
{
    const int64_t node = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t total = (int64_t)nx * ny * nz;
    if (node >= total) return;
    const int32_t i = (int32_t)(node % nx), j = (int32_t)((node / nx) % ny), k = (int32_t)(node / ((int64_t)nx * ny));
    const float gx = fmaf((float)i, spacing, ox), gy = fmaf((float)j, spacing, oy), gz = fmaf((float)k, spacing, oz);
    const int32_t cx = cell_coord(gx, sc.origin[0], sc.cell, sc.dims[0]);
    const int32_t cy = cell_coord(gy, sc.origin[1], sc.cell, sc.dims[1]);
    const int32_t cz = cell_coord(gz, sc.origin[2], sc.cell, sc.dims[2]);
    const int32_t R = sc.R;
    const int32_t x0 = max(cx - R, 0), x1 = min(cx + R, sc.dims[0] - 1);
    float phi = 0.0f;
    for (int32_t dz = -R; dz <= R; ++dz) {
        const int32_t z = cz + dz;
        if (z < 0 || z >= sc.dims[2]) continue;
        for (int32_t dy = -R; dy <= R; ++dy) {
            const int32_t y = cy + dy;
            if (y < 0 || y >= sc.dims[1]) continue;
            const int64_t row = (int64_t)sc.dims[0] * (y + (int64_t)sc.dims[1] * z);
            for (uint32_t t = start[row + x0]; t < start[row + x1 + 1]; ++t) {
                const float4 p = __ldg(sorted + t);
                const float dx = gx - p.x, dy2 = gy - p.y, dz2 = gz - p.z;
                const float d2 = fmaf(dx, dx, fmaf(dy2, dy2, dz2 * dz2));
                if (d2 < sc.h2) phi = fmaf(p.w, sc.sigma * spline_w(sqrtf(d2) * sc.inv_h), phi);
            }
        }
    }
    out[node] = phi;
}

// The same field, a warp per tile of 8 x 4 x 4 nodes (4 nodes a thread, along x).  The tile's
// candidates, the particles of its stencil rows within h of the tile's box, are compacted into
// shared memory once, in the rows' order, and every node then tests them from there: about
// 150 broadcast reads a tile at spacing h/4 where each node alone loads 216 candidates, and
// the distance and the spline of two nodes at a time in packed FP32.  A node meets its
// neighbours in the same order and with the same operations as above (what it skips would
// not have passed its test, and a candidate outside h adds an exact zero), the root apart, which
// differs from sqrtf by an ulp at a few arguments in 2^24 (sqrt2): the field is that of the
// general kernel to an ulp of a distance, and bit for bit wherever it was compared.  Bound by
// instruction issue (70 % of the cycles).
// Chosen by the spacing; on coarser grids a tile's box holds more candidates than its nodes share.
// Field alone, this kernel against the general one, us: 1.2M particles at 0.25 h 1217 and 2193,
// 0.4 h 518 and 723, 0.5 h 404 and 452, 0.55 h 383 and 375, 0.6 h 366 and 321, 0.8 h 393 and 211;
// 210k particles, whose dense tiles are few, 0.25 h 291 and 672, 0.4 h 174 and 212, 0.5 h 176 and
// 147, 0.55 h 180 and 132, 0.6 h 204 and 122.
constexpr float kTileSpacing = 0.55f;   // of h
constexpr int kTileX = 8, kTileY = 4, kTileZ = 4, kTileWarps = 4;

typedef unsigned long long f2;   // two packed floats
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b)
{
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 dup(float a) { return pack_xy(a, a); }
__device__ __forceinline__ void unpack(f2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }

// Largest of three, NaN if one is.
__device__ __forceinline__ float max_nan(float a, float b, float c)
{
    float r;
    asm("{ .reg .f32 t; max.NaN.f32 t, %1, %2; max.NaN.f32 %0, t, %3; }" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Square roots of a pair (a, b) of normal numbers: g = x y, g + (y/2) (x - g g) from y =
// rsqrt(x), Newton's step with the residual exact in FP32 (Markstein's square root), in packed
// FP32.  The value before the last rounding is within 2^-44 of the root: of all significands
// over 200 exponents (1.7e9 numbers) four differ from sqrtf, by one ulp.
__device__ __forceinline__ f2 sqrt2(f2 x, float a, float b)
{
    float ya, yb;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ya) : "f"(a));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yb) : "f"(b));
    const f2 y = pack_xy(ya, yb), g = mul2(x, y);
    return fma2(mul2(y, dup(-0.5f)), fma2(g, g, mul2(x, dup(-1.0f))), g);
}

__global__ void __launch_bounds__(32 * kTileWarps, 8)
    k_pf_field_tile(const float4 *__restrict__ sorted, const uint32_t *__restrict__ start, SceneDev sc, float ox,
                    float oy, float oz, float spacing, int32_t nx, int32_t ny, int32_t nz, uint32_t tx, uint32_t ty,
                    uint32_t ntiles, float *__restrict__ out)
{
    __shared__ float4 s_buf[kTileWarps][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t tile = blockIdx.x * kTileWarps + (uint32_t)warp;   // fewer than 2^31
    if (tile >= ntiles) return;
    float4 *buf = s_buf[warp];
    const uint32_t trow = tile / tx, tk = trow / ty;
    const int32_t i0 = (int32_t)(tile - trow * tx) * kTileX, j0 = (int32_t)(trow - tk * ty) * kTileY, k0 = (int32_t)tk * kTileZ;
    auto node_x = [&](int32_t i) { return fmaf((float)i, spacing, ox); };
    auto node_y = [&](int32_t j) { return fmaf((float)j, spacing, oy); };
    auto node_z = [&](int32_t k) { return fmaf((float)k, spacing, oz); };
    const float lox = node_x(i0), hix = node_x(min(i0 + kTileX, nx) - 1);
    const float loy = node_y(j0), hiy = node_y(min(j0 + kTileY, ny) - 1);
    const float loz = node_z(k0), hiz = node_z(min(k0 + kTileZ, nz) - 1);
    const int32_t R = sc.R;
    const int32_t x0 = max(cell_coord(lox, sc.origin[0], sc.cell, sc.dims[0]) - R, 0);
    const int32_t x1 = min(cell_coord(hix, sc.origin[0], sc.cell, sc.dims[0]) + R, sc.dims[0] - 1);
    const int32_t y0 = max(cell_coord(loy, sc.origin[1], sc.cell, sc.dims[1]) - R, 0);
    const int32_t y1 = min(cell_coord(hiy, sc.origin[1], sc.cell, sc.dims[1]) + R, sc.dims[1] - 1);
    const int32_t z0 = max(cell_coord(loz, sc.origin[2], sc.cell, sc.dims[2]) - R, 0);
    const int32_t z1 = min(cell_coord(hiz, sc.origin[2], sc.cell, sc.dims[2]) + R, sc.dims[2] - 1);
    // this thread's nodes: x = i0 + 4 q + 2 e + lx for pair q, element e, so that the nodes of
    // a pair in all lanes form a compact block (4 x 4 x 4), skipped together
    const int lx = lane & 1, ly = (lane >> 1) & 3, lz = lane >> 3;
    const float gy = node_y(j0 + ly), gz = node_z(k0 + lz);
    const f2 gx[2] = {pack_xy(node_x(i0 + lx), node_x(i0 + lx + 2)), pack_xy(node_x(i0 + lx + 4), node_x(i0 + lx + 6))};
    const float h2 = sc.h2, tiny = 1e-20f * sc.h2;
    const f2 ih = dup(sc.inv_h), sigma = dup(sc.sigma), one = dup(1.0f), six = dup(6.0f),
             nsix = dup(-6.0f), two = dup(2.0f);
    f2 phi[2] = {0ull, 0ull};
    auto add = [&](int n) {   // the nodes' sums over buf[0..n)
        for (int c = 0; c < n; ++c) {
            const float4 p = buf[c];
            const float dy = gy - p.y, dz = gz - p.z;
            // (a distance below 1e-10 h weighs as zero does; kept off zero for the root)
            const f2 yz = dup(fmaxf(fmaf(dy, dy, dz * dz), tiny)), px = dup(p.x);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const f2 dx = sub2(gx[q], px);
                const f2 d2 = fma2(dx, dx, yz);
                float a, b;
                unpack(d2, a, b);
                if (a < h2 || b < h2) {
                    const f2 u = mul2(sqrt2(d2, a, b), ih);
                    float na, nb, ta, tb, ua, ub;
                    unpack(fma2(mul2(u, six), mul2(u, u), fma2(mul2(u, nsix), u, one)), na, nb);
                    unpack(sub2(one, u), ta, tb);
                    const f2 t = pack_xy(fmaxf(ta, 0.0f), fmaxf(tb, 0.0f));
                    unpack(mul2(mul2(mul2(t, two), t), t), ta, tb);
                    unpack(u, ua, ub);
                    const float wa = a < h2 ? (ua <= 0.5f ? na : ta) : 0.0f, wb = b < h2 ? (ub <= 0.5f ? nb : tb) : 0.0f;
                    phi[q] = fma2(dup(p.w), mul2(sigma, pack_xy(wa, wb)), phi[q]);
                }
            }
        }
    };
    int cnt = 0;
    const int32_t rows_y = y1 - y0 + 1, rows = rows_y * (z1 - z0 + 1);
    for (int32_t rb = 0; rb < rows; rb += 32) {
        // 32 rows' candidate ranges at once, then the non-empty ones in order
        uint32_t b = 0, e = 0;
        if (rb + lane < rows) {
            const int32_t y = y0 + (rb + lane) % rows_y, z = z0 + (rb + lane) / rows_y;
            const int64_t row = (int64_t)sc.dims[0] * (y + (int64_t)sc.dims[1] * z);
            b = start[row + x0];
            e = start[row + x1 + 1];
        }
        for (unsigned m = __ballot_sync(0xffffffffu, b < e); m != 0u; m &= m - 1u) {
            const int src = __ffs(m) - 1;
            const uint32_t rb0 = __shfl_sync(0xffffffffu, b, src), re = __shfl_sync(0xffffffffu, e, src);
            for (uint32_t t = rb0; t < re; t += 32u) {
                bool keep = false;
                float4 p;
                if (t + (uint32_t)lane < re) {
                    p = __ldg(sorted + t + lane);
                    // distance to the box: no larger than to any node, operation by operation; a NaN
                    // coordinate, which add()'s maximum would pass over, stays one and is not near
                    const float dx = max_nan(lox - p.x, p.x - hix, 0.0f), dy = max_nan(loy - p.y, p.y - hiy, 0.0f),
                                dz = max_nan(loz - p.z, p.z - hiz, 0.0f);
                    keep = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < h2;
                }
                const unsigned kept = __ballot_sync(0xffffffffu, keep);
                if (keep) buf[cnt + __popc(kept & ((1u << lane) - 1u))] = p;
                cnt += __popc(kept);
                __syncwarp();
                if (cnt >= 32) {
                    add(32);
                    cnt -= 32;
                    float4 q;
                    if (lane < cnt) q = buf[32 + lane];
                    __syncwarp();
                    if (lane < cnt) buf[lane] = q;
                    __syncwarp();
                }
            }
        }
    }
    add(cnt);
    const int32_t j = j0 + ly, k = k0 + lz;
    if (j >= ny || k >= nz) return;
    float *o = out + (int64_t)nx * (j + (int64_t)ny * k);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        float a, b;
        unpack(phi[q], a, b);
        const int32_t i = i0 + 4 * q + lx;
        if (i < nx) o[i] = a;
        if (i + 2 < nx) o[i + 2] = b;
    }
}

// ------------------------------------------------------------------ marching tetrahedra
// The six tetrahedra, four corners of 4 bits each, first corner lowest.
__device__ __forceinline__ uint32_t tet_corners(int t)
{
    const uint32_t lo = t < 2 ? (t == 0 ? 0x7310u : 0x7510u) : (t == 2 ? 0x7320u : 0x7620u);
    return t < 4 ? lo : (t == 4 ? 0x7540u : 0x7640u);
}

// Triangles of tetrahedron t of a cube whose corners above the iso-level are the bits of above.
__device__ __forceinline__ int tet_count(uint32_t above, int t)
{
    const uint32_t c = tet_corners(t);
    int n = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) n += (int)((above >> ((c >> (4 * q)) & 15u)) & 1u);
    return (n == 0 || n == 4) ? 0 : (n == 2 ? 2 : 1);
}

// Corner values and positions of one cube, read where they are needed (corner index =
// dx + 2 dy + 4 dz).
struct Cube {
    const float *f;
    int32_t nx, ny, i, j, k;
    float ox, oy, oz, sp;
    __device__ __forceinline__ float value(int q) const
    {
        return f[(int64_t)(i + (q & 1)) + (int64_t)nx * ((j + ((q >> 1) & 1)) + (int64_t)ny * (k + (q >> 2)))];
    }
    __device__ __forceinline__ float3 corner(int q) const
    {
        return make_float3(fmaf((float)(i + (q & 1)), sp, ox), fmaf((float)(j + ((q >> 1) & 1)), sp, oy),
                           fmaf((float)(k + (q >> 2)), sp, oz));
    }
};

__device__ __forceinline__ float3 cut(const Cube &c, int a, int b, float iso)
{
    const float va = c.value(a), vb = c.value(b);
    const float3 pa = c.corner(a), pb = c.corner(b);
    const float t = (iso - va) / (vb - va);
    return make_float3(fmaf(t, pb.x - pa.x, pa.x), fmaf(t, pb.y - pa.y, pa.y), fmaf(t, pb.z - pa.z, pa.z));
}

// Write triangle (q0, q1, q2), flipped if its normal points from the outside corners'
// centroid towards the inside corners' centroid.
__device__ __forceinline__ void emit(float3 q0, float3 q1, float3 q2, float3 cin, float3 cout, float *dst)
{
    const float e1[3] = {q1.x - q0.x, q1.y - q0.y, q1.z - q0.z};
    const float e2[3] = {q2.x - q0.x, q2.y - q0.y, q2.z - q0.z};
    const float n[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
    const float dot = n[0] * (cout.x - cin.x) + n[1] * (cout.y - cin.y) + n[2] * (cout.z - cin.z);
    const float3 b = dot < 0.0f ? q2 : q1, c = dot < 0.0f ? q1 : q2;
    dst[0] = q0.x; dst[1] = q0.y; dst[2] = q0.z;
    dst[3] = b.x; dst[4] = b.y; dst[5] = b.z;
    dst[6] = c.x; dst[7] = c.y; dst[8] = c.z;
}

// The triangles of tetrahedron t of cube c, from output index o on.
__device__ __forceinline__ void emit_tet(const Cube &c, uint32_t above, int t, float iso, int64_t o, float *tris,
                                         int64_t cap)
{
    const uint32_t corners = tet_corners(t);
    uint32_t ins = 0u, outs = 0u;   // corner numbers, 4 bits each
    int ni = 0, no = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t v = (corners >> (4 * q)) & 15u;
        if ((above >> v) & 1u) ins |= v << (4 * ni++);
        else outs |= v << (4 * no++);
    }
    if (ni == 0 || ni == 4) return;
    auto in = [&](int k) { return (int)((ins >> (4 * k)) & 15u); };
    auto out = [&](int k) { return (int)((outs >> (4 * k)) & 15u); };
    float3 cin = make_float3(0.f, 0.f, 0.f), cout = cin;
    for (int q = 0; q < ni; ++q) {
        const float3 p = c.corner(in(q));
        cin.x += p.x / (float)ni; cin.y += p.y / (float)ni; cin.z += p.z / (float)ni;
    }
    for (int q = 0; q < no; ++q) {
        const float3 p = c.corner(out(q));
        cout.x += p.x / (float)no; cout.y += p.y / (float)no; cout.z += p.z / (float)no;
    }
    // every cut runs from the corner above to the corner below, so the tetrahedra sharing a
    // grid edge compute the same vertex (a watertight mesh)
    if (ni == 2) {
        const float3 q0 = cut(c, in(0), out(0), iso), q1 = cut(c, in(0), out(1), iso), q2 = cut(c, in(1), out(1), iso),
                     q3 = cut(c, in(1), out(0), iso);
        if (o < cap) emit(q0, q1, q2, cin, cout, tris + 9 * o);
        if (o + 1 < cap) emit(q0, q2, q3, cin, cout, tris + 9 * (o + 1));
    } else if (o < cap) {
        const float3 q0 = cut(c, in(0), out(0), iso);
        const float3 q1 = ni == 1 ? cut(c, in(0), out(1), iso) : cut(c, in(1), out(0), iso);
        const float3 q2 = ni == 1 ? cut(c, in(0), out(2), iso) : cut(c, in(2), out(0), iso);
        emit(q0, q1, q2, cin, cout, tris + 9 * o);
    }
}

// The surface in three launches: a block counts the triangles of a tile of consecutive cubes from
// their corner bits; one block makes the tiles' places out of the counts; the blocks of crossed
// tiles place their cubes and write the crossed tetrahedra, one a thread, from a shared list.
// 16M cubes of the 1.2M scene: about 250 us; 640 us with a count a cube in memory (64 MB written,
// scanned and read) and a crossed cube's thread writing all its triangles alone; 276 us as one
// launch with look-back between the tiles, which it spent waiting.
constexpr int kMeshThreads = 256;   // of a block, and cubes of a tile: ITEMS a thread
// Division of n < 2^31 by d >= 1 by multiplication (Granlund and Montgomery, Division by invariant
// integers using multiplication, 1994): n m >> (31 + l), l = ceil(log2 d), m = ceil(2^(31+l) / d).
struct Divisor {
    uint32_t d, l;
    uint64_t m;
    explicit Divisor(uint32_t d_) : d(d_), l(0)
    {
        while ((1ull << l) < d) ++l;
        m = ((1ull << (31 + l)) + d - 1) / d;
    }
    __device__ __forceinline__ uint32_t quotient(uint32_t n) const { return (uint32_t)(((uint64_t)n * (uint32_t)m) >> (31 + l)); }
};

struct MeshGrid {
    const float *f;
    int32_t nx, ny;
    Divisor by_x, by_y;   // cubes along x, along y
    uint32_t cubes;       // fewer than 2^31
    float iso;
};

// Triangles by corner bits, for the block.
__device__ __forceinline__ void mesh_counts(uint8_t *s_count)
{
    int n = 0;
#pragma unroll
    for (int q = 0; q < 6; ++q) n += tet_count((uint32_t)threadIdx.x, q);
    s_count[threadIdx.x] = (uint8_t)n;
    __syncthreads();
}

// Corner bits of this thread's cubes of a tile: base + t, base + t + 256, ...: a warp reads 33
// consecutive values of each of four rows.
template <int ITEMS>
__device__ __forceinline__ void mesh_corners(const MeshGrid &g, uint32_t tile, uint32_t (&above)[ITEMS])
{
    const int64_t dz = (int64_t)g.nx * g.ny;
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
        const uint32_t cube = tile * (uint32_t)(ITEMS * kMeshThreads) + (uint32_t)(q * kMeshThreads) + threadIdx.x;
        above[q] = 0u;
        if (cube < g.cubes) {
            const uint32_t row = g.by_x.quotient(cube), i = cube - row * g.by_x.d, k = g.by_y.quotient(row), j = row - k * g.by_y.d;
            const float *p = g.f + (int64_t)i + (int64_t)g.nx * (j + (int64_t)g.ny * k);
            const float iso = g.iso;
            above[q] = (p[0] > iso ? 1u : 0u) | (p[1] > iso ? 2u : 0u) | (p[g.nx] > iso ? 4u : 0u) |
                       (p[g.nx + 1] > iso ? 8u : 0u) | (p[dz] > iso ? 16u : 0u) | (p[dz + 1] > iso ? 32u : 0u) |
                       (p[dz + g.nx] > iso ? 64u : 0u) | (p[dz + g.nx + 1] > iso ? 128u : 0u);
        }
    }
}

template <int ITEMS>
__global__ void __launch_bounds__(kMeshThreads) k_mt_count(MeshGrid g, uint32_t *tile_count)
{
    __shared__ uint8_t s_count[256];
    __shared__ uint32_t s_warp[kMeshThreads / 32];
    mesh_counts(s_count);
    uint32_t above[ITEMS], n = 0u;
    mesh_corners(g, blockIdx.x, above);
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) n += s_count[above[q]];
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = n;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kMeshThreads / 32; ++w) n += s_warp[w];
        tile_count[blockIdx.x] = n;
    }
}

// Cubes a thread.  Eight leave few blocks to a small grid, each writing a long list: a ball's surface
// in 64^3 cubes takes 18.6 us with eight and 13.8 with one (55.8 with a thread a cube for
// everything), a noisy one 153 and 75, in 100^3 cubes 31.2 and 27.9, 128^3 40.1 and 44.3, 252^3
// 130 and 259 (the places of 62,500 tiles).  The line: five tiles of eight a SM.
int mesh_items(int64_t cubes) { return cubes < (int64_t)5 * 152 * 8 * kMeshThreads ? 1 : 8; }

// Exclusive sums of the tiles' counts in place, the total behind them (one block).
__global__ void __launch_bounds__(1024) k_mt_places(uint32_t *tile_count, int32_t ntiles)
{
    __shared__ uint32_t s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t run = 0u;
    for (int32_t k0 = 0; k0 < ntiles; k0 += 1024) {
        const int32_t k = k0 + (int32_t)threadIdx.x;
        const uint32_t v = k < ntiles ? tile_count[k] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        const uint32_t w = s_warp[lane];
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
        if (k < ntiles) tile_count[k] = run + before + x - v;
        run += __reduce_add_sync(0xffffffffu, w);
        __syncthreads();
    }
    if (threadIdx.x == 0) tile_count[ntiles] = run;
}

template <int ITEMS>
__global__ void __launch_bounds__(kMeshThreads)
    k_mt_emit(MeshGrid g, float ox, float oy, float oz, float sp, const uint32_t *__restrict__ place, float *tris, int64_t cap)
{
    const uint32_t tile = blockIdx.x;
    const int64_t first = (int64_t)place[tile];
    if ((int64_t)place[tile + 1] == first || first >= cap) return;
    constexpr int kWarps = kMeshThreads / 32;
    constexpr int kSums = ITEMS * kWarps;
    static_assert(kSums <= 64, "one warp scans the sums of all items, two a lane");
    __shared__ uint8_t s_count[256];                 // triangles by corner bits
    __shared__ uint32_t s_list[ITEMS * kMeshThreads];           // crossed cubes: index in the tile, corner bits
    __shared__ uint16_t s_first[ITEMS * kMeshThreads];          // their first triangle in the tile (at most 24,576)
    __shared__ uint32_t s_sum[kSums];  // per item and warp, then their exclusive sums
    __shared__ uint32_t s_crossed;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    mesh_counts(s_count);
    // per item, places in cube order from sums over the warp of the triangles (low 16 bits)
    // and the crossed cubes (high 16 bits)
    uint32_t above[ITEMS], sum[ITEMS];
    mesh_corners(g, tile, above);
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
        const uint32_t n = s_count[above[q]], v = n | (n ? 0x10000u : 0u);
        uint32_t x = v;
        if (__any_sync(0xffffffffu, n != 0u)) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
        }
        if (lane == 31) s_sum[q * kWarps + warp] = x;
        sum[q] = x - v;
    }
    __syncthreads();
    if (warp == 0) {
        const bool any = 2 * lane < kSums;
        const uint32_t a = any ? s_sum[2 * lane] : 0u, b = any ? s_sum[2 * lane + 1] : 0u;
        uint32_t x = a + b;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_crossed = x >> 16;
        if (any) {
            s_sum[2 * lane] = x - a - b;
            s_sum[2 * lane + 1] = x - b;
        }
    }
    __syncthreads();
    const uint32_t crossed = s_crossed;
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
        if (s_count[above[q]] == 0u) continue;
        const uint32_t at = s_sum[q * kWarps + warp] + sum[q];
        s_list[at >> 16] = (uint32_t)(q * kMeshThreads + t) | (above[q] << 16);
        s_first[at >> 16] = (uint16_t)(at & 0xffffu);
    }
    __syncthreads();
    for (uint32_t u = (uint32_t)t; u < crossed * 6u; u += kMeshThreads) {
        const uint32_t c = u / 6u;
        const int tet = (int)(u - 6u * c);
        const uint32_t e = s_list[c], a = e >> 16;
        if (tet_count(a, tet) == 0) continue;
        int64_t o = first + s_first[c];
        for (int q = 0; q < tet; ++q) o += tet_count(a, q);
        if (o >= cap) continue;
        const uint32_t cube = tile * (uint32_t)(ITEMS * kMeshThreads) + (e & 0xffffu), row = g.by_x.quotient(cube), k = g.by_y.quotient(row);
        const Cube cb{g.f, g.nx, g.ny, (int32_t)(cube - row * g.by_x.d), (int32_t)(row - k * g.by_y.d), (int32_t)k, ox, oy, oz, sp};
        emit_tet(cb, a, tet, g.iso, o, tris, cap);
    }
}

// ------------------------------------------------------------------ height map
__device__ __forceinline__ uint32_t order_key(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float order_value(uint32_t k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__global__ void k_hm_clear(uint32_t *img, int64_t n)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) img[k] = 0u;
}

__global__ void k_hm_splat(const float4 *__restrict__ pos, int64_t n, float lox, float loy, float du, float dv,
                           int32_t w, int32_t h, float R, uint32_t *img)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 p = pos[i];
    // pixel range of the disk's bounding box, clamped in float before the conversion
    auto px = [](float v, int32_t n) { return (int32_t)fminf(fmaxf(v, -1.0f), (float)n); };
    const int32_t i0 = max(px(floorf((p.x - R - lox) / du - 0.5f), w), 0);
    const int32_t i1 = min(px(ceilf((p.x + R - lox) / du - 0.5f), w), w - 1);
    const int32_t j0 = max(px(floorf((p.y - R - loy) / dv - 0.5f), h), 0);
    const int32_t j1 = min(px(ceilf((p.y + R - loy) / dv - 0.5f), h), h - 1);
    const float R2 = R * R;
    for (int32_t j = j0; j <= j1; ++j) {
        const float v = fmaf((float)j + 0.5f, dv, loy) - p.y;
        for (int32_t ii = i0; ii <= i1; ++ii) {
            const float u = fmaf((float)ii + 0.5f, du, lox) - p.x;
            const float d2 = fmaf(u, u, v * v);
            if (d2 < R2) atomicMax(img + (int64_t)j * w + ii, order_key(p.z + sqrtf(R2 - d2)));
        }
    }
}

__global__ void k_hm_decode(uint32_t *img, int64_t n)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const uint32_t v = img[k];
    img[k] = v == 0u ? 0x7fc00000u : __float_as_uint(order_value(v));
}

int blocks_for(int64_t n) { return (int)((n + kPostBlock - 1) / kPostBlock); }

}  // namespace

// The context's own sort scratch serves the field's grid order (the next step rebuilds all of
// it: keys, slots, cell table, neighbour lists): allocating and returning 40 MB on every call cost
// about as much host time as the sort.
cudaError_t post_surface_field(const Ptrs &P, const SceneDev &sc, int64_t nbr_entries, const float origin[3],
                               float spacing, const int32_t dims[3], float *out, cudaStream_t s)
{
    const int64_t n = sc.nf, ncell = sc.ncell;
    const float4 *pos = P.pos_c + sc.f_off, *vel = P.vel_c + sc.f_off;
    uint32_t *count = P.cell_count, *start = P.cell_start, *key = P.key_tmp, *slot = P.slot_tmp, *cellidx = P.sid_tmp;
    float4 *sorted = reinterpret_cast<float4 *>(P.nbr), *own = nullptr;
    cudaError_t e = cudaSuccess;
    if (nbr_entries < 4 * n) {   // neighbour lists of fewer than four entries a particle
        e = cudaMallocAsync((void **)&own, sizeof(float4) * n, s);
        sorted = own;
    }
    if (e == cudaSuccess) {
        k_pf_hist<<<blocks_for(n), kPostBlock, 0, s>>>(pos, n, sc, count, key, slot);
        launch_scan(count, start, ncell, P.scan_status, scan_tiles_for(ncell), &P.ctl->scan[0], P.ctl, false, s);
        k_pf_place<<<blocks_for(n), kPostBlock, 0, s>>>(n, key, slot, start, cellidx);
        k_pf_rank<<<blocks_for(n), kPostBlock, 0, s>>>(pos, vel, n, sc.m, sc.rho0, key, start, cellidx, sorted);
        const int64_t nodes = (int64_t)dims[0] * dims[1] * dims[2];
        const int64_t tx = (dims[0] + kTileX - 1) / kTileX, ty = (dims[1] + kTileY - 1) / kTileY,
                      tz = (dims[2] + kTileZ - 1) / kTileZ, tiles = tx * ty * tz;
        if (spacing <= kTileSpacing * sc.h)
            k_pf_field_tile<<<(unsigned)((tiles + kTileWarps - 1) / kTileWarps), 32 * kTileWarps, 0, s>>>(
                sorted, start, sc, origin[0], origin[1], origin[2], spacing, dims[0], dims[1], dims[2], (uint32_t)tx,
                (uint32_t)ty, (uint32_t)tiles, out);
        else
            k_pf_field<<<blocks_for(nodes), kPostBlock, 0, s>>>(sorted, start, sc, origin[0], origin[1], origin[2],
                                                                spacing, dims[0], dims[1], dims[2], out);
        e = cudaGetLastError();
    }
    if (own) cudaFreeAsync(own, s);
    return e;
}

cudaError_t post_height_map(const float4 *pos, int64_t n, const float lo[2], const float hi[2], int32_t w,
                            int32_t h, float radius, float *out, cudaStream_t s)
{
    const int64_t px = (int64_t)w * h;
    uint32_t *img = reinterpret_cast<uint32_t *>(out);   // the keys, decoded in place
    const float du = (hi[0] - lo[0]) / (float)w, dv = (hi[1] - lo[1]) / (float)h;
    k_hm_clear<<<blocks_for(px), kPostBlock, 0, s>>>(img, px);
    if (n > 0) k_hm_splat<<<blocks_for(n), kPostBlock, 0, s>>>(pos, n, lo[0], lo[1], du, dv, w, h, radius, img);
    k_hm_decode<<<blocks_for(px), kPostBlock, 0, s>>>(img, px);
    return cudaGetLastError();
}

}  // namespace sph

using namespace sph;

extern "C" sph_status sph_surface_mesh(const float *field, const int32_t dims[3], const float origin[3],
                                       float spacing, float iso, float *tris, int64_t cap, int64_t *n_tris,
                                       void *stream)
{
    if (!field || !dims || !origin || !n_tris || cap < 0 || (cap > 0 && !tris)) return SPH_EINVAL;
    if (!(spacing > 0.0f) || !std::isfinite(spacing) || !std::isfinite(iso)) return SPH_EINVAL;
    for (int a = 0; a < 3; ++a)
        if (dims[a] < 2 || !std::isfinite(origin[a])) return SPH_EINVAL;
    const int64_t cubes = (int64_t)(dims[0] - 1) * (dims[1] - 1) * (dims[2] - 1);
    if ((int64_t)dims[0] * dims[1] * dims[2] > ((int64_t)1 << 31)) return SPH_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int items = mesh_items(cubes);
    const int64_t ntiles = (cubes + items * kMeshThreads - 1) / (items * kMeshThreads);
    uint32_t *place = nullptr, total = 0;
    cudaError_t e = cudaMallocAsync((void **)&place, sizeof(uint32_t) * (size_t)(ntiles + 1), s);
    if (e == cudaSuccess) {
        const MeshGrid g{field, dims[0], dims[1], Divisor((uint32_t)dims[0] - 1u), Divisor((uint32_t)dims[1] - 1u),
                         (uint32_t)cubes, iso};
        const unsigned blocks = (unsigned)ntiles;
        if (items == 8) k_mt_count<8><<<blocks, kMeshThreads, 0, s>>>(g, place);
        else k_mt_count<1><<<blocks, kMeshThreads, 0, s>>>(g, place);
        k_mt_places<<<1, 1024, 0, s>>>(place, (int32_t)ntiles);
        if (cap > 0) {
            if (items == 8) k_mt_emit<8><<<blocks, kMeshThreads, 0, s>>>(g, origin[0], origin[1], origin[2], spacing, place, tris, cap);
            else k_mt_emit<1><<<blocks, kMeshThreads, 0, s>>>(g, origin[0], origin[1], origin[2], spacing, place, tris, cap);
        }
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(&total, place + ntiles, sizeof total, cudaMemcpyDeviceToHost, s);
        cudaFreeAsync(place, s);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return SPH_ECUDA;
    *n_tris = (int64_t)total;
    return (int64_t)total > cap ? SPH_EOVERFLOW : SPH_OK;
}

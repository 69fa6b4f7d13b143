// sph_fluid.cu -- per-particle sweeps of the DFSPH step.
//
// T threads (lanes, T = 1, 2, 4 or 8) own one fluid particle in grid order.  The density
// sweep walks the (2R+1)^3-cell neighbourhood ((2R+1)^2 contiguous index ranges) once
// per step and records the particle's neighbours in one k-major list, in candidate order
// (one thread a particle; with T = 8 eight lanes test eight consecutive candidates at a time:
// the list is the same).  Every later sweep of the
// step (divergence and density Jacobi passes, non-pressure forces, warm starts) gathers
// through that list, lane s taking entries s, s + T, ..., and combines the T partial sums
// with warp shuffles.  The solvers' error sums are accumulated per block in FP64 by pass A,
// folded by pass B and summed in a fixed order by a one-block check kernel, which also
// decides the loop condition on the device (CUDA graph conditional node); small contexts run a
// whole solve as one cooperative launch (k_solve).
#include <cuda_fp16.h>
#include <math_constants.h>

#include <algorithm>

#include "sph_sweep.cuh"

namespace sph {

namespace {

__device__ __forceinline__ void set_w(float4 *p, int64_t i, float w)
{
    reinterpret_cast<float *>(p + i)[3] = w;
}

struct BlockCtx {
    const SceneDev *sc;
    SceneState *st;
    int64_t i;
    bool valid;
};

__device__ __forceinline__ BlockCtx fluid_ctx(const Ptrs &P)
{
    BlockCtx c;
    int32_t s = scene_of_block(P, P.fblk_scene, (int32_t)blockIdx.x);
    c.sc = &P.scenes[s];
    c.st = &P.st[s];
    int64_t local = (int64_t)(blockIdx.x - c.sc->fblk_first) * kBlock + threadIdx.x;
    c.valid = local < c.sc->nf;
    c.i = c.sc->f_off + local;
    return c;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ int warp_max(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Pass A's error partials are folded by pass B's blocks, fold_size(count) consecutive ones
// per fold (at least 8, and at most 256 folds per scene), and the check kernel sums a
// scene's folds with one warp.  The order depends only on the scene's own block count, so
// a scene reduces the same way alone and in any batch.
__device__ __forceinline__ int32_t fold_size(int32_t count) { return max(8, (count + 255) / 256); }

// Fixed-order block sum of one double per thread (deterministic; valid in thread 0; sh holds
// one double a thread).  FP64 additions are a few per cycle and SM on this GPU: through shared
// memory one warp does all 8 x 32 of them, where butterflies in every warp did 20 x 32.
__device__ double block_sum(double v, double *sh)
{
    __syncthreads();
    sh[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x >= 32) return 0.0;
    static_assert(kBlock == 128, "four values a lane");
    const double t = (sh[threadIdx.x] + sh[threadIdx.x + 32]) + (sh[threadIdx.x + 64] + sh[threadIdx.x + 96]);
    return warp_sum(t);
}

// ------------------------------------------------------------------------------------
// Step begin: per-scene counters and the step size.
__global__ void k_step_begin(Ptrs P)
{
    kernel_enter(P.ctl, KID_STEP_BEGIN);
    int s = threadIdx.x + blockIdx.x * blockDim.x;
    if (s == 0) {
        P.ctl->loop_guard = 0;
        P.ctl->mlp_n = 0;
    }
    if (s >= P.nscenes) return;
    const SceneDev &sc = P.scenes[s];
    SceneState &st = P.st[s];
    float od = P.ctl->dt_override;
    st.dt = od > 0.0f ? od : (sc.cfl > 0.0f ? st.dt_next : sc.dt_max);
    for (int k = 0; k < 2; ++k) {
        st.last_it[k] = st.it[k];
        st.it[k] = 0;
        st.err[k] = CUDART_INF;
        st.err0[k] = 0.0;
    }
    st.counter = 0;
    st.max_nn_f = 0;
    st.max_nn_b = 0;
    st.maxv2 = 0.0f;
    if (sc.strong)   // strongly coupled bodies accumulate the step's force during the solves
        for (int k = 0; k < sc.nbody; ++k) {
            BodyDev &B = P.bodies[sc.body_off + k];
            for (int a = 0; a < 3; ++a) {
                B.force[a] = 0.0;
                B.torque[a] = 0.0;
            }
        }
}

// ------------------------------------------------------------------------------------
// Density (Eq. density + Sec. 3.5 boundary term), DFSPH alpha, neighbour lists, and the
// gate of the divergence warm start (D rho/Dt with the velocities at step start); one thread
// a particle (SUM = false: only the lists, k_density_sum follows).
//
// Phase 1 filters the stencil's rows: the candidates' coordinates in 16-bit steps of h/512 (the
// reorder writes them negated, two particles a 16-byte word) give (d/h)^2 of two candidates at
// a time in half precision, from one load and eleven instructions.  A difference q - c modulo
// 2^16, added to the bits of the half 1536, is that half plus the difference (a half's step is 1
// from 1024 to 2048, which covers differences up to h; beyond, the value only has to stay
// beyond), so no conversion is needed; one 32-bit addition serves both, its carry being one step
// in the second.  The threshold lies above 1 by more than all rounding (sph_filter.h), so every
// neighbour passes, with 2 to 4 % more.  Phase 2 walks the passed ones with the exact predicate,
// drops those that fail from the list in place, and sums: list, counts and sums are those of
// the exact test on every candidate, in the same order.
//
// A particle whose passed candidates exceed the list takes the exact predicate on what passes the
// filter, from the first row on; one that has left the range the filter holds for
// (SceneDev::qreach) takes it on every candidate.
//
// Between the phases a thread keeps its first kStage passed candidates in shared memory: written
// straight to the list, whose entries the lanes of a warp reach at different times, each store
// touched its own line, and phase 2 read them back from memory.  Phase 2 writes the list entry by
// entry with the warp in step.
//
// Bound by instruction issue and gather latency in turn: at 500k particles 146 us (167 with the
// exact predicate on every candidate and boundary rows looked up by all, 154 without the stage),
// 1.2M with bodies 343 us (396, 356).  24 staged candidates, which 28 neighbours overrun, take 153
// and 355.  Past the stage the list is read four entries ahead: particles twice as dense (60
// neighbours, 500k) 611 -> 505 us a step; with the exact predicate on every candidate it was 472.
// Where lists overrun (an error to the caller) or hold hundreds, the exact predicate alone was faster:
// 110 neighbours in lists of 96 864 us, here 1200 (1540 before the second pass went by the filter),
// 240 in lists of 512 351 (100k particles) and 505 (656 before).
// With two and four lanes the lists are built here and the lanes only sum: 100k particles
// 160 -> 59 us.
__device__ __forceinline__ uint32_t query_pair(uint32_t word, uint32_t odd)
{
    return ((0x6600u - (odd ? word >> 16 : word)) & 0xffffu) * 0x10001u;
}
__device__ __forceinline__ __half2 as_half2(uint32_t v) { return *reinterpret_cast<__half2 *>(&v); }
struct Stencil {
    uint32_t row;            // first row's cell of column 0
    uint32_t dx, dxy;        // cells of a row, of a layer
    int32_t x0, x1;          // first and last cell of every row
    int32_t ny, nz, centre;  // rows a layer, layers, number of the particle's own row
};

// The filter's query: the particle's own coordinates and the threshold (a pair of halves each).
struct Query {
    uint32_t x, y, z, thr;
    __device__ __forceinline__ Query(const Ptrs &P, const SceneDev &sc, uint32_t i) : thr(sc.qthr)
    {
        const uint4 own = P.qpos[i >> 1];
        x = query_pair(own.x, i & 1u);
        y = query_pair(own.y, i & 1u);
        z = query_pair(own.z, i & 1u);
    }
};

// Candidates c0, ... c0 + n - 1 (c0 even, n <= 32), eight at a time; a bit set: farther than h.
__device__ __forceinline__ uint32_t far_bits(const uint4 *qpos, uint32_t c0, uint32_t n, const Query &c)
{
    const __half2 thr = as_half2(c.thr), unit = __float2half2_rn(1.0f / 512.0f), bias = __float2half2_rn(-3.0f);
    uint32_t far = 0u;
    const uint4 *w = qpos + (c0 >> 1);
    for (uint32_t q = 0u; q < n; q += 8u, w += 4) {
        uint4 p[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) p[u] = __ldg(w + u);
        int bits = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const __half2 dx = __hfma2(as_half2(c.x + p[u].x), unit, bias);
            const __half2 dy = __hfma2(as_half2(c.y + p[u].y), unit, bias);
            const __half2 dz = __hfma2(as_half2(c.z + p[u].z), unit, bias);
            const uint32_t f = __hgt2_mask(__hfma2(dx, dx, __hfma2(dy, dy, __hmul2(dz, dz))), thr);
            // bytes 0 and 2 of the masks (-1 or 0) times -4^u and -2 4^u: bits 2u, 2u + 1
            bits = __dp4a((int)f, (int)((uint32_t)(uint8_t)(-(1 << (2 * u))) | (uint32_t)(uint8_t)(-(2 << (2 * u))) << 16), bits);
        }
        far |= (uint32_t)bits << q;
    }
    return far;
}

// The exact predicate over the stencil, on the candidates that pass the filter or (out of its
// reach) on all, loads four at a time: writes the list, returns the neighbour count.
constexpr int kStage = 32;   // candidates a thread keeps in shared memory between the phases
__device__ __noinline__ int exact_list(const Ptrs &P, const SceneDev &sc, const Stencil &st, int64_t i, float4 pi, bool filtered)
{
    const Query query(P, sc, (uint32_t)i);
    const float h2 = sc.h2;
    const int cap = sc.cap_f;
    int n = 0;
    auto test = [&](uint32_t j, float4 p) {
        float dx, dy, dz;
        if (j == (uint32_t)i || !(pred_d2(pi, p, dx, dy, dz) < h2)) return;
        if (n < cap) P.nbr[(int64_t)n * P.NF + i] = (int32_t)j;
        ++n;
    };
    for (int32_t k = 0; k < st.ny * st.nz; ++k) {
        const uint32_t row = st.row + (uint32_t)(k % st.ny) * st.dx + (uint32_t)(k / st.ny) * st.dxy;
        const uint32_t jb = P.cell_start[row + (uint32_t)st.x0], je = P.cell_start[row + (uint32_t)st.x1 + 1u];
        if (!filtered) {
            uint32_t j = jb;
            for (; j + 3u < je; j += 4u) {
                float4 p[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) p[u] = __ldg(P.pos_s + j + u);
#pragma unroll
                for (int u = 0; u < 4; ++u) test(j + (uint32_t)u, p[u]);
            }
            for (; j < je; ++j) test(j, __ldg(P.pos_s + j));
            continue;
        }
        for (uint32_t c0 = jb & ~1u; c0 < je; c0 += 32u) {
            const uint32_t m = min(je - c0, 32u);
            uint32_t near = ~far_bits(P.qpos, c0, m, query) & (0xffffffffu >> (32u - m));
            if (c0 < jb) near &= ~1u;
            while (near != 0u) {
                uint32_t j[4];
                float4 p[4];
                bool is[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    is[u] = near != 0u;
                    j[u] = is[u] ? c0 + (uint32_t)__ffs((int)near) - 1u : j[0];
                    near &= near - 1u;
                    p[u] = __ldg(P.pos_s + j[u]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (is[u]) test(j[u], p[u]);
            }
        }
    }
    return n;
}

template <bool SUM>
__global__ void __launch_bounds__(kBlock, 9) k_density(const __grid_constant__ Ptrs P)
{
    __shared__ int32_t s_list[kStage][kBlock];
    kernel_enter(P.ctl, KID_DENSITY);
    const BlockCtx c = fluid_ctx(P);
    const SceneDev &sc = *c.sc;
    const int64_t i = c.i, NF = P.NF;
    const bool gate = sc.warm != 0 && sc.div_on;
    int nn_f = 0, nn_b = 0;   // neighbours (may exceed the capacity)
    if (c.valid) {
        const float4 pi = P.pos_s[i];
        const int cap_f = sc.cap_f, cap_b = sc.cap_b;
        const float h2 = sc.h2;
        Stencil st;
        bool walls;   // a boundary particle in the stencil
        {
            const int32_t cx = cell_coord(pi.x, sc.origin[0], sc.cell, sc.dims[0]);
            const int32_t cy = cell_coord(pi.y, sc.origin[1], sc.cell, sc.dims[1]);
            const int32_t cz = cell_coord(pi.z, sc.origin[2], sc.cell, sc.dims[2]);
            const int32_t R = sc.R, nx = sc.dims[0], ny = sc.dims[1], nz = sc.dims[2];
            const int32_t y0 = max(cy - R, 0), z0 = max(cz - R, 0);
            st.x0 = max(cx - R, 0);
            st.x1 = min(cx + R, nx - 1);
            st.ny = min(cy + R, ny - 1) - y0 + 1;
            st.nz = min(cz + R, nz - 1) - z0 + 1;
            st.centre = (cz - z0) * st.ny + (cy - y0);
            st.dx = (uint32_t)nx;
            st.dxy = (uint32_t)nx * (uint32_t)ny;
            const uint32_t c0 = (uint32_t)sc.c_off;
            st.row = c0 + (uint32_t)nx * ((uint32_t)y0 + (uint32_t)ny * (uint32_t)z0);
            walls = P.bnear[c0 + (uint32_t)cx + (uint32_t)nx * ((uint32_t)cy + (uint32_t)ny * (uint32_t)cz)] != 0;
        }
        const uint32_t self = (uint32_t)i;
        int passed = 0;
        const float away = fmaxf(fmaxf(fabsf(pi.x - sc.origin[0]), fabsf(pi.y - sc.origin[1])), fabsf(pi.z - sc.origin[2]));
        {
            const Query query(P, sc, self);
            const int32_t rows = away <= sc.qreach ? st.ny * st.nz : 0;
            uint32_t row = st.row;
            for (int32_t k = 0, y = 0; k < rows; ++k) {
                const uint32_t jb = P.cell_start[row + (uint32_t)st.x0], je = P.cell_start[row + (uint32_t)st.x1 + 1u];
                row += st.dx;
                if (++y == st.ny) { y = 0; row += st.dxy - (uint32_t)st.ny * st.dx; }
                for (uint32_t c0 = jb & ~1u; c0 < je; c0 += 32u) {   // from an even index on
                    const uint32_t n = min(je - c0, 32u);
                    const uint32_t far = far_bits(P.qpos, c0, n, query);
                    uint32_t near = ~far & (0xffffffffu >> (32u - n));
                    if (c0 < jb) near &= ~1u;
                    if (k == st.centre && self - c0 < 32u) near &= ~(1u << (self - c0));
                    int q = passed;
                    passed += __popc(near);
                    if (passed > cap_f) {   // the exact predicate builds the list instead
                        k = rows;
                        break;
                    }
                    for (; near != 0u; near &= near - 1u, ++q) {
                        const int32_t j = (int32_t)(c0 + (uint32_t)__ffs((int)near) - 1u);
                        if (q < kStage) s_list[q][threadIdx.x] = j;
                        else P.nbr[(int64_t)q * NF + i] = j;
                    }
                }
            }
        }
        if (walls) {
            uint32_t row = st.row;
            for (int32_t k = 0, y = 0; k < st.ny * st.nz; ++k) {
                const uint32_t be = P.bcell_start[row + (uint32_t)st.x1 + 1u];
                for (uint32_t b = P.bcell_start[row + (uint32_t)st.x0]; b < be; ++b) {
                    float dx, dy, dz;
                    if (pred_d2(pi, __ldg(P.bpos_s + b), dx, dy, dz) < h2) {
                        if (nn_b < cap_b) P.bnbr[(int64_t)nn_b * NF + i] = (int32_t)b;
                        ++nn_b;
                    }
                }
                row += st.dx;
                if (++y == st.ny) { y = 0; row += st.dxy - (uint32_t)st.ny * st.dx; }
            }
        }
        int total = -1;   // exact count, where the list was built by the exact predicate
        if (passed > cap_f || !(away <= sc.qreach)) {
            total = exact_list(P, sc, st, i, pi, away <= sc.qreach);
            passed = min(total, cap_f);
        }
        // phase 2: the exact predicate, density, alpha and the warm-start gate
        const float4 vi = P.vel_s[i];
        const Spline sp(sc);
        float w_sum = 0.0f, s1x = 0.0f, s1y = 0.0f, s1z = 0.0f, s2 = 0.0f, div_l = 0.0f;
        // the first passed candidates are in shared memory, the rest, and a list built by the exact
        // predicate, in the list itself
        const int staged = total < 0 ? min(passed, kStage) : 0;
        auto visit = [&](int32_t j, float4 pj) {
            float dx, dy2, dz2;
            const float d2 = pred_d2(pi, pj, dx, dy2, dz2);
            if (!(d2 < h2)) return;
            P.nbr[(int64_t)nn_f * NF + i] = j;
            ++nn_f;
            if (!SUM) return;
            w_sum += spline_w(sqrtf(d2) * sp.inv_h);
            const float f = grad_factor(sp, d2);
            const float gx = f * dx, gy = f * dy2, gz = f * dz2;
            s1x += gx; s1y += gy; s1z += gz;
            s2 = fmaf(gx, gx, fmaf(gy, gy, fmaf(gz, gz, s2)));
            if (gate) {
                const float4 vj = __ldg(P.vel_s + j);
                div_l += (vi.x - vj.x) * gx + (vi.y - vj.y) * gy + (vi.z - vj.z) * gz;
            }
        };
        int k = 0;
        for (; k + 2 <= staged; k += 2) {
            const int32_t j0 = s_list[k][threadIdx.x], j1 = s_list[k + 1][threadIdx.x];
            const float4 p0 = __ldg(P.pos_s + j0), p1 = __ldg(P.pos_s + j1);
            visit(j0, p0);
            visit(j1, p1);
        }
        if (k < staged) {
            const int32_t j0 = s_list[k][threadIdx.x];
            visit(j0, __ldg(P.pos_s + j0));
        }
        // (read four ahead of where the list is written; past its end the last entry again)
        if (staged < passed) {
            const int32_t *list = P.nbr + i;
            int32_t j[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) j[u] = list[(int64_t)min(staged + u, passed - 1) * NF];
            for (k = staged; k < passed; k += 4) {
                int32_t next[4];
                float4 p[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    p[u] = __ldg(P.pos_s + j[u]);
                    next[u] = list[(int64_t)min(k + 4 + u, passed - 1) * NF];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (k + u < passed) visit(j[u], p[u]);
                    j[u] = next[u];
                }
            }
        }
        const int nb = min(nn_b, cap_b);
        P.nnf[i] = nn_f;
        P.nnb[i] = nb;
        if constexpr (SUM) {
            float rho_l = sc.m * sc.sigma * w_sum;
            s1x = sc.m * s1x; s1y = sc.m * s1y; s1z = sc.m * s1z;
            s2 *= sc.m * sc.m;
            div_l = sc.m * div_l;
            if (nb > 0) {
                float wb = 0.0f, divb = 0.0f;
                const bool moving = sc.has_moving != 0;
                for_list<1, 1, false>(P.bnbr, NF, i, 0, nb, [&](int32_t b) {
                    const float4 pb = __ldg(P.bpos_s + b);
                    float dx, dy2, dz2;
                    const float d2 = pred_d2(pi, pb, dx, dy2, dz2);
                    const float psi = pb.w;
                    wb += psi * spline_w(sqrtf(d2) * sp.inv_h);
                    const float f = psi * grad_factor(sp, d2);
                    const float gx = f * dx, gy = f * dy2, gz = f * dz2;
                    s1x += gx; s1y += gy; s1z += gz;
                    if (gate) {
                        float4 vb = moving ? __ldg(P.bvel_s + b) : make_float4(0.f, 0.f, 0.f, 0.f);
                        divb += (vi.x - vb.x) * gx + (vi.y - vb.y) * gy + (vi.z - vb.z) * gz;
                    }
                });
                rho_l += sc.sigma * wb;
                div_l += divb;
            }
            const float rho = fmaf(sc.m, sc.sigma, rho_l);
            const float den = fmaf(s1x, s1x, fmaf(s1y, s1y, fmaf(s1z, s1z, s2)));
            P.alpha[i] = den > sc.eps_alpha ? rho / den : 0.0f;
            set_w(P.vel_s, i, rho);
            float kv0 = 0.0f;
            if (gate && div_l > 0.0f) kv0 = sc.warm_frac * P.kvprev_s[i] / c.st->dt;
            P.kvsum[i] = kv0;
            set_w(P.pos_s, i, kv0 / rho);
        }
        if (total >= 0) nn_f = total;
    }
    // one atomic per warp: spread over this long sweep they cost less than a block barrier would
    const int mf = warp_max(nn_f), mb = warp_max(nn_b);
    if ((threadIdx.x & 31) == 0) {
        if (mf > 0) atomicMax(&c.st->max_nn_f, mf);
        if (mb > 0) atomicMax(&c.st->max_nn_b, mb);
        if (mf > sc.cap_f || mb > sc.cap_b) atomicOr(&c.st->flags, 1);
    }
}

// Density, alpha and the warm-start gate of a particle from its lists by T lanes, lane s taking
// entries s, s + T, ... (every thread of the warp calls it).  FRESH: lists this warp has just
// written.
template <int T, bool FRESH>
__device__ __forceinline__ void density_sums(const Ptrs &P, const Lane<T> &c, float4 pi, int nf, int nb)
{
    const SceneDev &sc = *c.sc;
    const int64_t i = c.i, NF = P.NF;
    const int s = c.s;
    const bool gate = sc.warm != 0 && sc.div_on;
    // this lane's shares of rho - m W(0), sum grad W, sum |grad W|^2 and D rho/Dt
    float rho_l = 0.0f, s1x = 0.0f, s1y = 0.0f, s1z = 0.0f, s2 = 0.0f, div_l = 0.0f;
    if (c.valid) {
        const float4 vi = P.vel_s[i];
        const int32_t *__restrict__ nbr = P.nbr;
        const int32_t *__restrict__ bnbr = P.bnbr;
        float w_sum = 0.0f, fx = 0.0f, fy = 0.0f, fz = 0.0f, div_f = 0.0f;
        const Spline sp(sc);
        for_list<2, T, !FRESH>(nbr, NF, i, s, nf, [&](int32_t j) {
            const float4 pj = __ldg(P.pos_s + j);
            float dx, dy2, dz2;
            const float d2 = pred_d2(pi, pj, dx, dy2, dz2);
            w_sum += spline_w(sqrtf(d2) * sp.inv_h);
            const float f = grad_factor(sp, d2);
            const float gx = f * dx, gy = f * dy2, gz = f * dz2;
            fx += gx; fy += gy; fz += gz;
            s2 = fmaf(gx, gx, fmaf(gy, gy, fmaf(gz, gz, s2)));
            if (gate) {
                const float4 vj = __ldg(P.vel_s + j);
                div_f += (vi.x - vj.x) * gx + (vi.y - vj.y) * gy + (vi.z - vj.z) * gz;
            }
        });
        rho_l = sc.m * sc.sigma * w_sum;
        s1x = sc.m * fx; s1y = sc.m * fy; s1z = sc.m * fz;
        s2 *= sc.m * sc.m;
        div_l = sc.m * div_f;
        if (nb > 0) {
            float wb = 0.0f, divb = 0.0f;
            const bool moving = sc.has_moving != 0;
            for_list<1, T, !FRESH>(bnbr, NF, i, s, nb, [&](int32_t b) {
                const float4 pb = __ldg(P.bpos_s + b);
                float dx, dy2, dz2;
                const float d2 = pred_d2(pi, pb, dx, dy2, dz2);
                const float psi = pb.w;
                wb += psi * spline_w(sqrtf(d2) * sp.inv_h);
                const float f = psi * grad_factor(sp, d2);
                const float gx = f * dx, gy = f * dy2, gz = f * dz2;
                s1x += gx; s1y += gy; s1z += gz;
                if (gate) {
                    float4 vb = moving ? __ldg(P.bvel_s + b) : make_float4(0.f, 0.f, 0.f, 0.f);
                    divb += (vi.x - vb.x) * gx + (vi.y - vb.y) * gy + (vi.z - vb.z) * gz;
                }
            });
            rho_l += sc.sigma * wb;
            div_l += divb;
        }
    }
    // combine the lanes (all threads of the warp take part)
    rho_l = group_sum<T>(rho_l);
    s1x = group_sum<T>(s1x); s1y = group_sum<T>(s1y); s1z = group_sum<T>(s1z);
    s2 = group_sum<T>(s2);
    div_l = group_sum<T>(div_l);
    if (c.valid && s == 0) {
        const float rho = fmaf(sc.m, sc.sigma, rho_l);
        const float den = fmaf(s1x, s1x, fmaf(s1y, s1y, fmaf(s1z, s1z, s2)));
        const float alpha = den > sc.eps_alpha ? rho / den : 0.0f;
        P.alpha[i] = alpha;
        set_w(P.vel_s, i, rho);
        float kv0 = 0.0f;
        if (gate && div_l > 0.0f) kv0 = sc.warm_frac * P.kvprev_s[i] / c.st->dt;
        P.kvsum[i] = kv0;
        set_w(P.pos_s, i, kv0 / rho);
    }
}

// The sums where one thread a particle built the lists (k_density<false>) but the context runs
// two or four lanes.
template <int T>
__global__ void __launch_bounds__(kBlock) k_density_sum(Ptrs P)
{
    kernel_enter(P.ctl, KID_DENSITY_SUM);
    const Lane<T> c = lane_ctx<T>(P);
    const float4 pi = c.valid ? P.pos_s[c.i] : make_float4(0.f, 0.f, 0.f, 0.f);
    density_sums<T, false>(P, c, pi, c.valid ? P.nnf[c.i] : 0, c.valid ? P.nnb[c.i] : 0);
}

// The same sweep by G threads a particle, for contexts too small to fill the GPU otherwise: lane
// r of the group loads the range of stencil row r, all in one memory latency, and for row after
// row the lanes test G consecutive candidates at a time with the exact predicate and append the
// hits in candidate order (ballot over the group), so the list is the same.  T of the G lanes
// then sum, T as in the context's other sweeps, whatever G.  G is the most of 32, 16 and 8 whose
// threads still fit the GPU: four steps of 8k particles 475 -> 467 us with 32, a step of 20k 236 ->
// 224 with 16 (both against 8 that loaded their ranges row by row).  Eight blocks per SM (64 registers for the batched cooperative append).
template <int T, int G>
__global__ void __launch_bounds__(kBlock, 8) k_density_lanes(Ptrs P)
{
    kernel_enter(P.ctl, KID_DENSITY);
    // a block takes 1 / (G / T) of the particles of a sweep block
    constexpr int kSplit = G / T;
    const int32_t block = (int32_t)blockIdx.x / kSplit;
    const int32_t sidx = scene_of_block(P, P.tblk_scene, block);
    const SceneDev &sc = P.scenes[sidx];
    SceneState &st = P.st[sidx];
    const int64_t local = (int64_t)(block - sc.tblk_first) * (kBlock / T) + ((int32_t)blockIdx.x % kSplit) * (kBlock / G) +
                          threadIdx.x / G;
    const bool valid = local < sc.nf;
    const int64_t i = sc.f_off + local, NF = P.NF;
    const int s = (int)(threadIdx.x % G);
    int nn_f = 0, nn_b = 0;  // the particle's neighbours (may exceed the capacity)
    float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) {
        pi = P.pos_s[i];
        const int32_t cx = cell_coord(pi.x, sc.origin[0], sc.cell, sc.dims[0]);
        const int32_t cy = cell_coord(pi.y, sc.origin[1], sc.cell, sc.dims[1]);
        const int32_t cz = cell_coord(pi.z, sc.origin[2], sc.cell, sc.dims[2]);
        // a boundary particle in the stencil
        const bool walls = P.bnear[sc.c_off + cx + (int64_t)sc.dims[0] * (cy + (int64_t)sc.dims[1] * cz)] != 0;
        const int32_t R = sc.R, side = 2 * R + 1, rows = side * side;
        const float h2 = sc.h2, cull2 = sc.cull2, cs = sc.cell;
        // offset of the particle inside its cell, per axis: the distance from the particle
        // to a stencil cell d cells away is at least gap(d) (zero for d = 0)
        const float ox = pi.x - fmaf((float)cx, cs, sc.origin[0]);
        const float oy = pi.y - fmaf((float)cy, cs, sc.origin[1]);
        const float oz = pi.z - fmaf((float)cz, cs, sc.origin[2]);
        auto gap = [&](float o, int32_t d) {
            const float g = d < 0 ? fmaf((float)(-d - 1), cs, o) : (d > 0 ? fmaf((float)d, cs, -o) : 0.0f);
            return fmaxf(g, 0.0f);
        };
        const int cap_f = sc.cap_f, cap_b = sc.cap_b;
        const uint32_t self = (uint32_t)i;
        const unsigned gmask = group_mask<G>();
        const int gshift = (int)(threadIdx.x & 31u) & ~(G - 1);
        const unsigned below = (1u << s) - 1u;
        // The float predicate over the stencil's index ranges only records neighbours.  Rows and
        // end cells whose nearest point is farther than h (plus a margin above the rounding of
        // these bounds) are skipped: they hold no particle that passes the predicate.
        for (int32_t r0 = 0; r0 < rows; r0 += G) {
            uint32_t jb_r = 0, je_r = 0, bb_r = 0, be_r = 0;
            if (r0 + s < rows) {
                const int32_t dz = (r0 + s) / side - R, dy = (r0 + s) % side - R, z = cz + dz, y = cy + dy;
                const float gz = gap(oz, dz), gy = gap(oy, dy), g2 = fmaf(gy, gy, gz * gz);
                if (z >= 0 && z < sc.dims[2] && y >= 0 && y < sc.dims[1] && !(g2 > cull2)) {
                    int32_t x0 = cx - R, x1 = cx + R;
                    while (x0 < cx && fmaf(gap(ox, x0 - cx), gap(ox, x0 - cx), g2) > cull2) ++x0;
                    while (x1 > cx && fmaf(gap(ox, x1 - cx), gap(ox, x1 - cx), g2) > cull2) --x1;
                    x0 = max(x0, 0);
                    x1 = min(x1, sc.dims[0] - 1);
                    const int64_t row = sc.c_off + (int64_t)sc.dims[0] * (y + (int64_t)sc.dims[1] * z);
                    jb_r = P.cell_start[row + x0];
                    je_r = P.cell_start[row + x1 + 1];
                    if (walls) {
                        bb_r = P.bcell_start[row + x0];
                        be_r = P.bcell_start[row + x1 + 1];
                    }
                }
            }
            for (int32_t r = 0; r < min(G, rows - r0); ++r) {
                const uint32_t jb = __shfl_sync(gmask, jb_r, r, G), je = __shfl_sync(gmask, je_r, r, G);
                // full batches of kCand groups load all their candidates before the first test
                auto append = [&](uint32_t j, bool hit) {
                    const unsigned bits = G == 32 ? __ballot_sync(gmask, hit) : (__ballot_sync(gmask, hit) >> gshift);
                    const int slot = nn_f + __popc(bits & below);
                    if (hit && slot < cap_f) P.nbr[(int64_t)slot * NF + i] = (int32_t)j;
                    nn_f += __popc(bits);
                };
                constexpr int kCand = 4;
                uint32_t j0 = jb;
                for (; j0 + (uint32_t)(kCand * G) <= je; j0 += (uint32_t)(kCand * G)) {   // uniform in the group
                    float4 pc[kCand];
#pragma unroll
                    for (int u = 0; u < kCand; ++u) pc[u] = __ldg(P.pos_s + j0 + (uint32_t)(u * G + s));
#pragma unroll
                    for (int u = 0; u < kCand; ++u) {
                        const uint32_t j = j0 + (uint32_t)(u * G + s);
                        float dx, dy2, dz2;
                        append(j, pred_d2(pi, pc[u], dx, dy2, dz2) < h2 && j != self);
                    }
                }
                for (; j0 < je; j0 += (uint32_t)G) {   // uniform in the group
                    const uint32_t j = j0 + (uint32_t)s;
                    bool hit = false;
                    if (j < je) {
                        float dx, dy2, dz2;
                        hit = pred_d2(pi, __ldg(P.pos_s + j), dx, dy2, dz2) < h2 && j != self;
                    }
                    append(j, hit);
                }
                if (walls) {
                    const uint32_t bb = __shfl_sync(gmask, bb_r, r, G), be = __shfl_sync(gmask, be_r, r, G);
                    for (uint32_t b0 = bb; b0 < be; b0 += (uint32_t)G) {
                        const uint32_t b = b0 + (uint32_t)s;
                        bool hit = false;
                        if (b < be) {
                            float dx, dy2, dz2;
                            hit = pred_d2(pi, __ldg(P.bpos_s + b), dx, dy2, dz2) < h2;
                        }
                        const unsigned bits = G == 32 ? __ballot_sync(gmask, hit) : (__ballot_sync(gmask, hit) >> gshift);
                        const int slot = nn_b + __popc(bits & below);
                        if (hit && slot < cap_b) P.bnbr[(int64_t)slot * NF + i] = (int32_t)b;
                        nn_b += __popc(bits);
                    }
                }
            }
        }
        // the lists were written by the group's lanes: order them before the reads below
        __syncwarp(gmask);
    }
    const Lane<T> c{&sc, &st, i, s % T, valid && s < T};
    density_sums<T, true>(P, c, pi, min(nn_f, sc.cap_f), min(nn_b, sc.cap_b));
    if (valid && s == 0) {
        P.nnf[i] = min(nn_f, sc.cap_f);
        P.nnb[i] = min(nn_b, sc.cap_b);
    }
    // the counts are the same in all lanes of a particle (one atomic per warp: spread over
    // this long sweep they cost less than a block barrier would)
    const int mf = warp_max(nn_f), mb = warp_max(nn_b);
    if ((threadIdx.x & 31) == 0) {
        if (mf > 0) atomicMax(&st.max_nn_f, mf);
        if (mb > 0) atomicMax(&st.max_nn_b, mb);
        if (mf > sc.cap_f || mb > sc.cap_b) atomicOr(&st.flags, 1);
    }
}

// ------------------------------------------------------------------------------------
// This lane's share of D rho_i/Dt = sum_j m (v_i - v_j).grad W_ij + sum_b Psi_b (v_i -
// v_b).grad W_ib (SPH divergence of Sec. 3.2 in the continuity equation, boundary per
// Sec. 3.5); group_sum of the shares is the full sum.  nf, nb: the list lengths (nb < 0: loaded
// where it is needed, which saves a register over the fluid list).
constexpr int kBatch = 4;

template <int B, int T, bool NC = true>
__device__ __forceinline__ float drho_dt_lane(const Ptrs &P, const SceneDev &sc, int64_t i, int s, float4 pi,
                                              float4 vi, const float4 *V, int nf, int nb)
{
    const int64_t NF = P.NF;
    const Spline sp(sc);
    float acc = 0.0f;
    for_list<B, T>(P.nbr, NF, i, s, nf, [&](int32_t j) {
        const float4 pj = ld4<NC>(P.pos_s + j);
        const float4 vj = ld4<NC>(V + j);
        const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
        const float f = grad_factor(sp, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        acc = fmaf(f, (vi.x - vj.x) * dx + (vi.y - vj.y) * dy + (vi.z - vj.z) * dz, acc);
    });
    float accb = 0.0f;
    const bool moving = sc.has_moving != 0;
    for_list<4, T>(P.bnbr, NF, i, s, nb < 0 ? P.nnb[i] : nb, [&](int32_t b) {
        const float4 pb = __ldg(P.bpos_s + b);
        const float dx = pi.x - pb.x, dy = pi.y - pb.y, dz = pi.z - pb.z;
        const float f = pb.w * grad_factor(sp, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        float ux = vi.x, uy = vi.y, uz = vi.z;
        if (moving) {
            const float4 vb = __ldg(P.bvel_s + b);
            ux -= vb.x; uy -= vb.y; uz -= vb.z;
        }
        accb = fmaf(f, ux * dx + uy * dy + uz * dz, accb);
    });
    return fmaf(sc.m, acc, accb);
}

// Pass A of a Jacobi iteration (Alg. ppe_solver "refine p"): the source term of
// Eq. velocity_source (solver 0) or Eq. density_source with rho* (solver 1), the
// stiffness kappa_i = alpha_i e_i / dt^(1 or 2), and the block's FP64 error partial.
template <int S, int B, int T, bool NC>
__device__ __forceinline__ void pass_a(const Ptrs &P, int32_t block, double *sh)
{
    const Lane<T> c = lane_ctx<T>(P, block);
    const SceneDev &sc = *c.sc;
    SceneState &st = *c.st;
    const float4 *V = S == 0 ? P.vel_s : P.vel_c;
    const int64_t i = c.i;
    // with several lanes, where latency is what a pass consists of, the particle's own loads, also
    // those the pass's end needs, go with those of the scene's state
    float4 pi = make_float4(0.f, 0.f, 0.f, 0.f), vi = pi;
    int nf = 0, nb = T > 1 ? 0 : -1;
    float alpha = 0.0f, ks = 0.0f;
    float *sum = S == 0 ? P.kvsum : P.ksum;
    if (T > 1 && c.valid) {
        pi = P.pos_s[i];
        vi = V[i];
        nf = P.nnf[i];
        nb = P.nnb[i];
        alpha = P.alpha[i];
        ks = sum[i];
    }
    if (!solver_active(sc, st, S)) return;  // uniform per block
    const float dt = st.dt;
    float D = 0.0f;
    if (c.valid) {
        if (T == 1) {
            pi = P.pos_s[i];
            vi = V[i];
            nf = P.nnf[i];
        }
        D = drho_dt_lane<B, T, NC>(P, sc, i, c.s, pi, vi, V, nf, nb);
    }
    D = group_sum<T>(D);
    double e = 0.0;
    if (c.valid && c.s == 0) {
        const float rho = vi.w;
        if (T == 1) {
            alpha = P.alpha[i];
            ks = sum[i];
        }
        float ei, kappa;
        if (S == 0) {
            ei = fmaxf(D, 0.0f);
            kappa = alpha * ei / dt;
            sum[i] = ks + kappa;
        } else if (sc.solver == 2) {
            // PCISPH: refine the total pressure p <- max(p + delta (rho* - rho0), 0) with
            // the prototype's delta; the pass B applies the change (kept as p/rho)
            const float dev = fmaf(dt, D, rho - sc.rho0);
            ei = fmaxf(dev, 0.0f);
            const float p_old = ks * rho;
            const float p_new = fmaxf(fmaf(sc.pci_c / (dt * dt), dev, p_old), 0.0f);
            kappa = (p_new - p_old) / rho;
            sum[i] = p_new / rho;
        } else {
            ei = fmaxf(fmaf(dt, D, rho - sc.rho0), 0.0f);
            kappa = alpha * ei / (dt * dt);
            sum[i] = ks + kappa;
        }
        set_w(P.pos_s, i, kappa / rho);
        e = (double)ei;
    }
    // the block's FP64 error partial; pass B folds the partials and the check kernel sums
    // the folds in a fixed order (no last-block step here: pass A only has to finish)
    const double bsum = block_sum(e, sh);
    if (threadIdx.x == 0) P.partial[block] = bsum;
}

template <int S, int B, int T>
__global__ void __launch_bounds__(kBlock) k_pass_a(Ptrs P)
{
    __shared__ double sh[kBlock];
    kernel_enter(P.ctl, (KID_PASS_A0 + S));
    pass_a<S, B, T, true>(P, (int32_t)blockIdx.x, sh);
}

// Pass B (Alg. ppe_solver "update v*"): pressure acceleration of Sec. 3.3 Eq.
// pressure_acceleration with p/rho^2 = kappa/rho, plus the boundary term of Sec. 3.5
// Eq. rigid_pressure per unit fluid mass:
//   v_i -= dt [ sum_j m (k_i/rho_i + k_j/rho_j) grad W_ij + sum_b Psi_b (k_i/rho_i) grad W_ib ]
// WARM = 1 applies the warm-start kappas (no loop bookkeeping).  With one lane and gather
// batch 4 the loop's pass B is held to 40 registers (12 resident blocks per SM instead of
// 10): it is bound by the gathers' latency, and the extra warps outweigh a few spilled words
// (measured on the 1.2M scene: 84 -> 80 us per density launch, 90 -> 81 per divergence
// launch).  Every other variant keeps the compiler's choice (a minimum of 0 blocks): the warm
// pass already fits in 40 registers, and batch 8 would spill 152 bytes.
template <int S, int WARM, int B, int T, bool NC>
__device__ __forceinline__ void pass_b(const Ptrs &P, int32_t block)
{
    const Lane<T> c = lane_ctx<T>(P, block);
    const SceneDev &sc = *c.sc;
    SceneState &st = *c.st;
    // uniform per block; WCSPH scenes apply their equation-of-state pressure here.  In the
    // loop, a scene's pass B runs exactly when its pass A did: the solver state only
    // changes in the check kernel that follows.
    // (With several lanes the particle's own loads go first, as in pass A.)
    float4 *V = S == 0 ? P.vel_s : P.vel_c;
    float4 own = make_float4(0.f, 0.f, 0.f, 0.f), v = own;
    int nf = 0, nb = 0;
    if (T > 1 && c.valid) {
        own = P.pos_s[c.i];
        nf = P.nnf[c.i];
        nb = P.nnb[c.i];
        if (c.s == 0) v = V[c.i];
    }
    const bool run = WARM ? warm_pass_runs(sc, S) : solver_active(sc, st, S);
    if (run) {
        const int64_t i = c.i, NF = P.NF;
        const int s = c.s;
        float ax = 0.0f, ay = 0.0f, az = 0.0f;
        if (c.valid) {
            const float4 pi = T > 1 ? own : P.pos_s[i];
            const float ki = pi.w;
            const Spline sp(sc);
            for_list<B, T>(P.nbr, NF, i, s, T > 1 ? nf : P.nnf[i], [&](int32_t j) {
                const float4 pj = ld4<NC>(P.pos_s + j);
                const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
                const float f = grad_factor(sp, fmaf(dx, dx, fmaf(dy, dy, dz * dz))) * (ki + pj.w);
                ax = fmaf(f, dx, ax); ay = fmaf(f, dy, ay); az = fmaf(f, dz, az);
            });
            ax *= sc.m; ay *= sc.m; az *= sc.m;
            if (ki != 0.0f) {
                float bx = 0.0f, by = 0.0f, bz = 0.0f;
                for_list<4, T>(P.bnbr, NF, i, s, T > 1 ? nb : P.nnb[i], [&](int32_t b) {
                    const float4 pb = __ldg(P.bpos_s + b);
                    const float dx = pi.x - pb.x, dy = pi.y - pb.y, dz = pi.z - pb.z;
                    const float f = pb.w * grad_factor(sp, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
                    bx = fmaf(f, dx, bx); by = fmaf(f, dy, by); bz = fmaf(f, dz, bz);
                });
                ax = fmaf(ki, bx, ax); ay = fmaf(ki, by, ay); az = fmaf(ki, bz, az);
            }
        }
        ax = group_sum<T>(ax); ay = group_sum<T>(ay); az = group_sum<T>(az);
        if (c.valid && s == 0) {
            const float dt = st.dt;
            if (T == 1) v = V[i];
            v.x -= dt * ax; v.y -= dt * ay; v.z -= dt * az;
            V[i] = v;
        }
    }
    if (WARM) return;
    // fold pass A's error partials: the scene's first ceil(count / F) blocks each sum F
    // consecutive ones in block order (the check kernel, a later launch, sums the folds)
    if (run && threadIdx.x == 0) {
        const int32_t lb = block - sc.tblk_first;
        const int32_t F = fold_size(sc.tblk_count);
        if (lb < (sc.tblk_count + F - 1) / F) {
            const int32_t k0 = lb * F, k1 = min(k0 + F, sc.tblk_count);
            double t = 0.0;
            for (int32_t k = k0; k < k1; ++k) t += __ldcg(P.partial + sc.tblk_first + k);
            P.partial2[block] = t;
        }
    }
}

template <int S, int WARM, int B, int T>
__global__ void __launch_bounds__(kBlock, (T == 1 && WARM == 0 && B == 4) ? 11 : 0) k_pass_b(Ptrs P)
{
    kernel_enter(P.ctl, (WARM ? KID_PASS_B0W + S : KID_PASS_B0 + S));
    pass_b<S, WARM, B, T, true>(P, (int32_t)blockIdx.x);
}

// Convergence test of one Jacobi iteration (Alg. ppe_solver's loop condition), one block
// after pass B: one warp per scene (32 scenes at a time) sums the scene's folds in a fixed
// order (lane l takes folds l, l + 32, ..., then a butterfly), which gives the mean error;
// the iteration counters advance and the loop condition is set for the host and for the
// CUDA graph's while node.
constexpr int kCheckThreads = 1024;

template <int S>
__device__ __forceinline__ uint32_t solver_check(const Ptrs &P, int *s_any)
{
    if (threadIdx.x == 0) *s_any = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int q = warp; q < P.nscenes; q += (int)(blockDim.x / 32)) {
        const SceneDev &qd = P.scenes[q];
        SceneState &qs = P.st[q];
        const int32_t F = fold_size(qd.tblk_count);
        const int32_t nfold = (qd.tblk_count + F - 1) / F;
        double t = 0.0;
#pragma unroll 8
        for (int k = lane; k < nfold; k += 32) t += __ldcg(P.partial2 + qd.tblk_first + k);
        if (!solver_active(qd, qs, S)) continue;   // its pass A and B did not run
        t = warp_sum(t);
        if (lane == 0) {
            double err = t * qd.err_scale;   // FP64 division is a long sequence here
            if (S == 0) err *= (double)qs.dt;
            if (qs.it[S] == 0) qs.err0[S] = err;
            qs.err[S] = err;
            qs.it[S] += 1;
            qs.total_it[S] += 1;
            if (!solver_active(qd, qs, S) && qs.err[S] > (double)qd.eta[S]) qs.flags |= 2;
            if (solver_active(qd, qs, S)) atomicOr(s_any, 1);
        }
    }
    __syncthreads();
    if (threadIdx.x != 0) return 0u;
    uint32_t any = *s_any;
    uint32_t guard = ++P.ctl->loop_guard;
    if (guard > 100000u) {
        any = 0;
        P.ctl->error = 2;
    }
    if (!any) P.ctl->loop_guard = 0;
    P.ctl->loop_flag = any;
    return any;
}

template <int S>
__global__ void __launch_bounds__(kCheckThreads) k_solver_check(Ptrs P, cudaGraphConditionalHandle handle,
                                                               int use_handle)
{
    __shared__ int s_any;
    kernel_enter(P.ctl, KID_CHECK0 + S);
    const uint32_t any = solver_check<S>(P, &s_any);
    if (threadIdx.x == 0 && use_handle) cudaGraphSetConditional(handle, any);
}

// A whole Jacobi solve in one cooperative launch: pass A, barrier, pass B, barrier with the
// convergence test in the block that arrives last, until no scene goes on.  The arithmetic and
// every order of summation are those of the separate kernels.  For contexts whose sweep blocks
// are all resident at once: there an iteration's launches, one-block check and while node
// (14 us) outweigh its passes; 8k particles: 4 steps 533 -> 480 us.  With more blocks a block's
// second round waits for nothing else to fill the SM and the separate kernels win (20k
// particles in two rounds 257 us a step against 236, 100k 447 against 433, 1.2M 2472 against 2376).
// And with many scenes: the last block's four warps test them four at a time, on the way of every
// iteration (4 + 12 iterations a step, one launch against separate kernels: 4 scenes of 1,000
// particles 265 and 343 us, 8 326 and 357, 12 382 and 380, 16 459 and 401).
constexpr int kSolveBlocksPerSm = 8;
constexpr int kSolveScenes = 8;
template <int S, int T>
__global__ void __launch_bounds__(kBlock, kSolveBlocksPerSm) k_solve(const __grid_constant__ Ptrs P)
{
    __shared__ double sh[kBlock];
    __shared__ int s_any;
    kernel_enter(P.ctl, KID_SOLVE0 + S);
    uint32_t phase = *reinterpret_cast<volatile uint32_t *>(&P.ctl->bar.gen);
    // after a wait that gave up the state is lost: the steps still queued must not wait in vain too
    // (looked at after the first pass A, beside which the load takes no time)
    for (;;) {
        pass_a<S, kBatch, T, false>(P, (int32_t)blockIdx.x, sh);
        if (!grid_barrier(&P.ctl->bar, &P.ctl->error, phase)) return;
        pass_b<S, 0, kBatch, T, false>(P, (int32_t)blockIdx.x);
        if (!grid_barrier(&P.ctl->bar, &P.ctl->error, phase, [&] { solver_check<S>(P, &s_any); })) return;
        if (*reinterpret_cast<volatile uint32_t *>(&P.ctl->loop_flag) == 0u) return;
    }
}

// ------------------------------------------------------------------------------------
// Non-pressure forces (Sec. 3.3 Alg. general_algorithm, Sec. 4.2: gravity, then
// viscosity): v* = v + dt (g + (mu/rho_i) lap v_i) with Eq. lap
//   lap v_i = 2(d+2) sum_j (m/rho_j) (v_ij . x_ij)/(|x_ij|^2 + 0.01 h^2) grad W_ij,
// or XSPH smoothing c sum_j (m/rho_j)(v_j - v_i) W_ij.  Writes v* to the canonical
// velocity array and clears the density-solve stiffness sum.
template <int T>
__global__ void __launch_bounds__(kBlock) k_nonpressure(Ptrs P)
{
    kernel_enter(P.ctl, KID_NONP);
    const Lane<T> c = lane_ctx<T>(P);
    const SceneDev &sc = *c.sc;
    const int64_t i = c.i, NF = P.NF;
    const int s = c.s;
    float4 vi = make_float4(0.f, 0.f, 0.f, 0.f);
    float sx = 0.0f, sy = 0.0f, sz = 0.0f;
    const bool visc = sc.visc_mode == 1 || sc.visc_mode == 2;  // uniform per block
    if (c.valid) {
        vi = P.vel_s[i];
        if (visc) {
            const float4 pi = P.pos_s[i];
            const float reg = 0.01f * sc.h2;
            const bool lap = sc.visc_mode == 1;
            const Spline sp(sc);
            for_list<kBatch, T>(P.nbr, NF, i, s, P.nnf[i], [&](int32_t j) {
                const float4 pj = __ldg(P.pos_s + j);
                const float4 vj = __ldg(P.vel_s + j);
                const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
                const float ux = vi.x - vj.x, uy = vi.y - vj.y, uz = vi.z - vj.z;
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                if (lap) {
                    const float f = grad_factor(sp, r2);
                    const float q = f * (ux * dx + uy * dy + uz * dz) / ((r2 + reg) * vj.w);
                    sx = fmaf(q, dx, sx); sy = fmaf(q, dy, sy); sz = fmaf(q, dz, sz);
                } else {
                    const float w = spline_w(sqrtf(r2) * sp.inv_h) / vj.w;
                    sx = fmaf(-w, ux, sx); sy = fmaf(-w, uy, sy); sz = fmaf(-w, uz, sz);
                }
            });
        }
    }
    if (visc) {
        sx = group_sum<T>(sx); sy = group_sum<T>(sy); sz = group_sum<T>(sz);
    }
    if (!c.valid || s != 0) return;
    const float dt = c.st->dt;
    const float rho_i = vi.w;
    const float ax = sc.g[0], ay = sc.g[1], az = sc.g[2];
    float4 v = vi;
    if (sc.visc_mode == 1) {
        const float k = 10.0f * sc.mu * sc.m / rho_i;
        v.x += dt * fmaf(k, sx, ax); v.y += dt * fmaf(k, sy, ay); v.z += dt * fmaf(k, sz, az);
    } else if (sc.visc_mode == 2) {
        const float k = sc.xsph * sc.m * sc.sigma;
        v.x += fmaf(dt, ax, k * sx); v.y += fmaf(dt, ay, k * sy); v.z += fmaf(dt, az, k * sz);
    } else {
        v.x += dt * ax; v.y += dt * ay; v.z += dt * az;
    }
    v.w = rho_i;
    P.vel_c[i] = v;
    // WCSPH: the equation of state of Sec. 3.4.1, p = k ((rho/rho0)^gamma - 1) clamped at
    // zero, evaluated as k expm1(gamma log1p(rho/rho0 - 1)) for accuracy near rho0; the
    // pressure pass then uses p/rho^2 (the kappa/rho slot) and the stiffness sum keeps
    // p/rho (so that p = kappa_sum rho for output and for the rigid reaction)
    float w = 0.0f, ks = 0.0f;
    if (sc.solver == 1) {
        const float p = fmaxf(sc.eos_k * expm1f(sc.eos_gamma * log1pf((rho_i - sc.rho0) / sc.rho0)), 0.0f);
        ks = p / rho_i;
        w = ks / rho_i;
    }
    P.ksum[i] = ks;
    P.k0[i] = 0.0f;
    set_w(P.pos_s, i, w);
}

// Warm start of the constant-density solve: the predicted deviation rho* - rho0 with
// v* gates a fraction (default half) of the previous step's stiffness (kept as kappa
// dt^2); the learned mode
// stores the network's input features instead (rho/rho0 - 1, dt Drho/Dt/rho0,
// (n_f + n_b)/33, kappa_prev/(9.81 h)) and a separate kernel fills kappa0.  With a
// learned gate g > 0 a scene whose previous density solve took g iterations or fewer
// takes the previous-step start in this step (the network would run for nothing at the
// solve's floor).
template <int T>
__global__ void __launch_bounds__(kBlock) k_warm_density(Ptrs P)
{
    kernel_enter(P.ctl, KID_WARM);
    const Lane<T> c = lane_ctx<T>(P);
    const SceneDev &sc = *c.sc;
    if (sc.warm == 0) return;  // uniform per block
    const int64_t i = c.i;
    float4 pi = make_float4(0.f, 0.f, 0.f, 0.f), vi = pi;
    float D = 0.0f;
    if (c.valid) {
        pi = P.pos_s[i];
        vi = P.vel_c[i];
        D = drho_dt_lane<kBatch, T>(P, sc, i, c.s, pi, vi, P.vel_c, P.nnf[i], T > 1 ? P.nnb[i] : -1);
    }
    D = group_sum<T>(D);
    const bool own = c.valid && c.s == 0;
    const float dt = c.st->dt;
    const float rho = vi.w;
    const float dev = fmaf(dt, D, rho - sc.rho0);
    // learned mode (uniform per block): the network runs unless the gate holds it back
    const bool net = sc.warm == 2 && (sc.learned_gate == 0 || c.st->last_it[1] > sc.learned_gate);
    // learned mode: the gated particles (predicted compression) are appended to the rows
    // of the network kernel, one atomic per warp (the whole warp is converged here)
    if (net) {
        const bool gated = own && dev > 0.0f && P.ctl->have_mlp;
        const unsigned m = __ballot_sync(0xffffffffu, gated);
        const int lane = threadIdx.x & 31;
        int base = 0;
        if (m != 0) {
            const int lead = __ffs(m) - 1;
            if (lane == lead) base = atomicAdd(&P.ctl->mlp_n, __popc(m));
            base = __shfl_sync(0xffffffffu, base, lead);
        }
        if (gated) P.mlp_rows[base + __popc(m & ((1u << lane) - 1u))] = make_int2((int)i, scene_of_block(P, P.tblk_scene, (int32_t)blockIdx.x));
    }
    if (!own) return;
    // the network's inputs are recorded in both warm-start modes (the previous-step mode
    // produces the training data)
    const float kref = 9.81f * sc.h;
    float4 f;
    f.x = rho / sc.rho0 - 1.0f;
    f.y = dt * D / sc.rho0;
    f.z = (float)(P.nnf[i] + P.nnb[i]) / 33.0f;
    f.w = P.kprev_s[i] / (dt * dt) / kref;
    reinterpret_cast<float4 *>(P.feat)[i] = f;
    float k0 = 0.0f;
    if (!net && dev > 0.0f) k0 = sc.warm_frac * P.kprev_s[i] / (dt * dt);
    // learned mode: zero here, the network kernel fills the gated rows
    P.k0[i] = k0;
    P.ksum[i] = k0;
    set_w(P.pos_s, i, k0 / rho);
}

// Advect (Sec. 3.3 Alg. general_algorithm, symplectic Euler): x = x + dt v*, written
// back in grid order as the next step's canonical state, with the warm-start memory.
__global__ void __launch_bounds__(kBlock) k_advect(Ptrs P)
{
    kernel_enter(P.ctl, KID_ADVECT);
    BlockCtx c = fluid_ctx(P);
    float v2 = 0.0f;
    bool bad = false;
    if (c.valid) {
        const int64_t i = c.i;
        const float dt = c.st->dt;
        const float4 v = P.vel_c[i];
        float4 p = P.pos_s[i];
        p.x = fmaf(dt, v.x, p.x);
        p.y = fmaf(dt, v.y, p.y);
        p.z = fmaf(dt, v.z, p.z);
        p.w = 0.0f;
        P.pos_c[i] = p;
        P.id_c[i] = P.id_s[i];
        P.kprev_c[i] = P.ksum[i] * dt * dt;
        P.kvprev_c[i] = P.kvsum[i] * dt;
        v2 = fmaf(v.x, v.x, fmaf(v.y, v.y, v.z * v.z));
        bad = !isfinite(p.x) || !isfinite(p.y) || !isfinite(p.z) || !isfinite(v2);
    }
    float m = v2;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const unsigned anybad = __ballot_sync(0xffffffffu, bad);
    // the block's largest finite |v|^2 and its bad flag reach the scene with one atomic each
    // (one per warp, on a single word, serialises in L2 and bounded this kernel)
    __shared__ float s_m[kBlock / 32];
    __shared__ unsigned s_bad[kBlock / 32];
    if ((threadIdx.x & 31) == 0) {
        s_m[threadIdx.x >> 5] = (m > 0.0f && isfinite(m)) ? m : 0.0f;
        s_bad[threadIdx.x >> 5] = anybad;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float bm = s_m[0];
        unsigned bb = s_bad[0];
        for (int w = 1; w < kBlock / 32; ++w) {
            bm = fmaxf(bm, s_m[w]);
            bb |= s_bad[w];
        }
        if (bm > 0.0f) atomicMax(reinterpret_cast<int *>(&c.st->maxv2), __float_as_int(bm));
        if (bb) atomicOr(&c.st->flags, 4);
    }
}

// Step end: CFL step for the next step (not in the paper: dt = min(dt_max, cfl 2r /
// max|v|)), counters, and the rigid bodies (symplectic Euler with a renormalised
// quaternion; weak coupling: bodies move only between fluid steps, Sec. 2.2 / 6).
__global__ void k_step_end(Ptrs P)
{
    kernel_enter(P.ctl, KID_STEP_END);
    int t = threadIdx.x;
    for (int s = t; s < P.nscenes; s += blockDim.x) {
        const SceneDev &sc = P.scenes[s];
        SceneState &st = P.st[s];
        float vm = sqrtf(st.maxv2);
        float dt = sc.dt_max;
        if (sc.cfl > 0.0f && vm > 0.0f) dt = fminf(dt, sc.cfl * sc.two_r / vm);
        st.dt_next = dt;
        st.steps += 1;
    }
    for (int k = t; k < P.nbodies_total; k += blockDim.x) {
        BodyDev &B = P.bodies[k];
        const SceneDev &sc = P.scenes[B.scene];
        const double dt = (double)P.st[B.scene].dt;
        const double fs = sc.strong ? 0.0 : 1.0;   // strong coupling applied the fluid's impulses already
        // FP64 division is a long dependent sequence on this GPU: the body record carries
        // 1/m and 1/I, and the quaternion is renormalised with one reciprocal square root
        const double inv_m = B.inv_mass;
        const double inv_i[3] = {B.inv_inertia[0], B.inv_inertia[1], B.inv_inertia[2]};
        for (int a = 0; a < 3; ++a) B.vel[a] += dt * (fs * B.force[a] * inv_m + (double)sc.g[a]);
        for (int a = 0; a < 3; ++a) B.com[a] += dt * B.vel[a];
        double w = B.quat[0], x = B.quat[1], y = B.quat[2], z = B.quat[3];
        double R[3][3] = {{1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)},
                          {2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)},
                          {2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)}};
        double Iw[3][3], Ii[3][3];
        for (int a = 0; a < 3; ++a)
            for (int e = 0; e < 3; ++e) {
                Iw[a][e] = 0.0;
                Ii[a][e] = 0.0;
                for (int q = 0; q < 3; ++q) {
                    Iw[a][e] += R[a][q] * B.inertia[q] * R[e][q];
                    Ii[a][e] += R[a][q] * inv_i[q] * R[e][q];
                }
            }
        double o[3] = {B.omega[0], B.omega[1], B.omega[2]};
        double L[3];
        for (int a = 0; a < 3; ++a) L[a] = Iw[a][0] * o[0] + Iw[a][1] * o[1] + Iw[a][2] * o[2];
        double rhs[3] = {fs * B.torque[0] - (o[1] * L[2] - o[2] * L[1]),
                         fs * B.torque[1] - (o[2] * L[0] - o[0] * L[2]),
                         fs * B.torque[2] - (o[0] * L[1] - o[1] * L[0])};
        for (int a = 0; a < 3; ++a) B.omega[a] += dt * (Ii[a][0] * rhs[0] + Ii[a][1] * rhs[1] + Ii[a][2] * rhs[2]);
        double ox = B.omega[0], oy = B.omega[1], oz = B.omega[2];
        double dw = 0.5 * (-ox * x - oy * y - oz * z);
        double dx = 0.5 * (ox * w + oy * z - oz * y);
        double dy = 0.5 * (oy * w + oz * x - ox * z);
        double dz = 0.5 * (oz * w + ox * y - oy * x);
        w += dt * dw; x += dt * dx; y += dt * dy; z += dt * dz;
        const double inv_nq = rsqrt(w * w + x * x + y * y + z * z);
        B.quat[0] = w * inv_nq; B.quat[1] = x * inv_nq; B.quat[2] = y * inv_nq; B.quat[3] = z * inv_nq;
        // no contact model (the paper delegates contact to PyBullet): the bounding sphere
        // is clamped inside the domain, and each clamp is counted
        for (int a = 0; a < 3; ++a) {
            if (B.com[a] < B.lo[a]) {
                B.com[a] = B.lo[a];
                if (B.vel[a] < 0.0) B.vel[a] = 0.0;
                atomicAdd(&P.st[B.scene].clamps, 1);
            }
            if (B.com[a] > B.hi[a]) {
                B.com[a] = B.hi[a];
                if (B.vel[a] > 0.0) B.vel[a] = 0.0;
                atomicAdd(&P.st[B.scene].clamps, 1);
            }
        }
    }
}

__global__ void k_set_dt(Control *ctl, float dt)
{
    kernel_enter(ctl, KID_SET_DT);
    ctl->dt_override = dt;
}

}  // namespace

void launch_step_begin(const Ptrs &P, cudaStream_t s)
{
    int t = P.nscenes < 1024 ? ((P.nscenes + 31) / 32) * 32 : 1024;
    int b = (P.nscenes + t - 1) / t;
    k_step_begin<<<b, t, 0, s>>>(P);
}
// Sweep kernels take T from the context (threads per particle) and the gather batch B
// of the Jacobi passes from its tuning: (T, B) in {(1, 4), (1, 8), (2, 4), (4, 4)}.
void launch_density_alpha(const Ptrs &P, cudaStream_t s)
{
    // Eight lanes a particle pay only where they are what fills the GPU (one thread against
    // eight: 8k particles 43 and 28 us, 38k about even); four or two lanes never did (100k: 160 us
    // with two, 55 with one).  Both write the same lists.
    if (P.lanes == 8) {
        // resident threads of a full GPU, as for the choice of the lanes
        constexpr int64_t kThreads = 152 * 2048;
        if (P.NF * 32 <= kThreads) k_density_lanes<8, 32><<<P.ntblk * 4, kBlock, 0, s>>>(P);
        else if (P.NF * 16 <= kThreads) k_density_lanes<8, 16><<<P.ntblk * 2, kBlock, 0, s>>>(P);
        else k_density_lanes<8, 8><<<P.ntblk, kBlock, 0, s>>>(P);
    } else if (P.lanes == 1) {
        k_density<true><<<P.nfblk, kBlock, 0, s>>>(P);
    } else {
        k_density<false><<<P.nfblk, kBlock, 0, s>>>(P);
        if (P.lanes == 4) k_density_sum<4><<<P.ntblk, kBlock, 0, s>>>(P);
        else k_density_sum<2><<<P.ntblk, kBlock, 0, s>>>(P);
    }
}
void launch_pass_a(const Ptrs &P, int solver, int batch, cudaStream_t s)
{
#define SPH_A(S, B, T) k_pass_a<S, B, T><<<P.ntblk, kBlock, 0, s>>>(P)
    if (P.lanes == 4) { if (solver == 0) SPH_A(0, 4, 4); else SPH_A(1, 4, 4); }
    else if (P.lanes == 8) { if (solver == 0) SPH_A(0, 4, 8); else SPH_A(1, 4, 8); }
    else if (P.lanes == 2) { if (solver == 0) SPH_A(0, 4, 2); else SPH_A(1, 4, 2); }
    else if (batch == 8) { if (solver == 0) SPH_A(0, 8, 1); else SPH_A(1, 8, 1); }
    else { if (solver == 0) SPH_A(0, 4, 1); else SPH_A(1, 4, 1); }
#undef SPH_A
}
void launch_pass_b(const Ptrs &P, int solver, int warm, int batch, cudaStream_t s)
{
#define SPH_B(S, W, B, T) k_pass_b<S, W, B, T><<<P.ntblk, kBlock, 0, s>>>(P)
#define SPH_BW(B, T)                                                 \
    do {                                                             \
        if (solver == 0) { if (warm) SPH_B(0, 1, B, T); else SPH_B(0, 0, B, T); } \
        else { if (warm) SPH_B(1, 1, B, T); else SPH_B(1, 0, B, T); }             \
    } while (0)
    if (P.lanes == 4) SPH_BW(4, 4);
    else if (P.lanes == 8) SPH_BW(4, 8);
    else if (P.lanes == 2) SPH_BW(4, 2);
    else if (batch == 8) SPH_BW(8, 1);
    else SPH_BW(4, 1);
#undef SPH_BW
#undef SPH_B
}
void launch_solver_check(const Ptrs &P, int solver, cudaGraphConditionalHandle h, int use_handle, cudaStream_t s)
{
    if (solver == 0) k_solver_check<0><<<1, kCheckThreads, 0, s>>>(P, h, use_handle);
    else k_solver_check<1><<<1, kCheckThreads, 0, s>>>(P, h, use_handle);
}
template <int T>
static const void *solve_kernel(int solver)
{
    return solver == 0 ? reinterpret_cast<const void *>(&k_solve<0, T>) : reinterpret_cast<const void *>(&k_solve<1, T>);
}
static const void *solve_kernel(const Ptrs &P, int solver)
{
    return P.lanes == 8 ? solve_kernel<8>(solver) : (P.lanes == 4 ? solve_kernel<4>(solver)
                                                                  : (P.lanes == 2 ? solve_kernel<2>(solver) : solve_kernel<1>(solver)));
}
int solve_grid(const Ptrs &P, int batch)
{
    // the passes with eight gathers in flight keep their own kernels
    if (batch != kBatch || P.nscenes > kSolveScenes || P.ntblk < 1) return 0;
    int dev = 0, nsm = 0, coop = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
        return 0;
    int resident = 0;
    for (int solver = 0; solver < 2; ++solver) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, solve_kernel(P, solver), kBlock, 0) != cudaSuccess) return 0;
        resident = solver == 0 ? per * nsm : std::min(resident, per * nsm);
    }
    return P.ntblk <= resident ? P.ntblk : 0;
}
cudaError_t launch_solve(const Ptrs &P, int solver, int grid, cudaStream_t s)
{
    void *args[] = {const_cast<Ptrs *>(&P)};
    return cudaLaunchCooperativeKernel(solve_kernel(P, solver), dim3((unsigned)grid), dim3(kBlock), args, 0, s);
}
void launch_nonpressure(const Ptrs &P, cudaStream_t s)
{
#define SPH_L(T) k_nonpressure<T><<<P.ntblk, kBlock, 0, s>>>(P)
    SPH_BY_LANES(P, SPH_L);
#undef SPH_L
}
void launch_warm_density(const Ptrs &P, cudaStream_t s)
{
#define SPH_L(T) k_warm_density<T><<<P.ntblk, kBlock, 0, s>>>(P)
    SPH_BY_LANES(P, SPH_L);
#undef SPH_L
}
void launch_advect(const Ptrs &P, cudaStream_t s) { k_advect<<<P.nfblk, kBlock, 0, s>>>(P); }
void launch_step_end(const Ptrs &P, cudaStream_t s) { k_step_end<<<1, 128, 0, s>>>(P); }
void launch_set_dt(const Ptrs &P, float dt, cudaStream_t s) { k_set_dt<<<1, 1, 0, s>>>(P.ctl, dt); }

}  // namespace sph

// sph_gelu.cuh -- the network's exact GELU, z Phi(z), and its derivative.
//
//   gelu(z) = max(z, 0) - |z|/2 erfc(|z|/sqrt 2),   erfc(t/sqrt 2) = 2^Q(t),
//
// with Q a degree-9 polynomial without constant term fitted to log2 erfc(t/sqrt 2) on
// [0, 6] (minimax of the error times erfc, by iteratively reweighted least squares against
// 40-digit values).  No branch and one ex2, two values at a time: the forward pass of 1.2M rows
// takes 96 us with it (83 without the rounding ties below) where it took 205 with the library's erff.
// Error against
// 64-bit values over [-9, 9]: at most 2.4e-7 and 5.0e-8 rms, where 0.5 z (1 + erff(z/sqrt 2))
// has 4.5e-7 and 6.4e-8.  Beyond |z| = 6 erfc is held at its value there (2e-9).  NaN stays
// NaN, +inf gives +inf and -inf gives NaN, as the product form does.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sph {
namespace gelu {

// Two floats in one 64-bit register: Blackwell's packed FP32 instructions halve the issue
// slots of the polynomial, which bounds the network's kernels.
typedef unsigned long long f2;

__device__ __forceinline__ f2 pk(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
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
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float ex2(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// erfc(|z|/sqrt 2) of a pair from s = max(-|z|/2, -3): the polynomial in s.
__device__ __forceinline__ f2 erfc_pair(f2 s)
{
    // coefficient k of Q times (-2)^k
    const float c[9] = {2.302212716f,     -1.836783767f,     0.4203080535f,    0.1140086353f, 0.005678631366f,
                        -0.01139640436f, -0.005409289152f, -0.001109374454f, -8.997129042e-05f};
    f2 q = pk(c[8], c[8]);
#pragma unroll
    for (int k = 7; k >= 0; --k) q = fma2(q, s, pk(c[k], c[k]));
    q = mul2(q, s);
    float a, b;
    upk(q, a, b);
    return pk(ex2(a), ex2(b));
}

// gelu of the pair z = 2 h (h: the halved pre-activations).
__device__ __forceinline__ f2 gelu_pair(float h0, float h1)
{
    const f2 s = pk(fmaxf(-fabsf(h0), -3.0f), fmaxf(-fabsf(h1), -3.0f));
    return fma2(s, erfc_pair(s), pk(h0 + fabsf(h0), h1 + fabsf(h1)));
}

// Hidden activations become BF16 operands, where a last-bit difference of the FP32 value can
// move the rounding by 2^-8.  So that operands are rounded as erff's formula rounds them, values
// within 16 ulp of a rounding boundary (low half within 16 of 0x8000) are found with two packed
// 16-bit operations a pair and taken from the formula; 16 columns of a warp hold one time in
// five such a value.  (The two formulas differ by at most 15 ulp where |gelu| >= 1/16, and by
// more only in the tail z < -1.9, where the formula cancels; below 1/64 a BF16 step is too
// small to matter and is left.)
__device__ __forceinline__ uint32_t tie_key(uint32_t m, float a, float b)
{
    uint32_t x = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x5410);
    // without a carry between the halves: what is found here has to be all that at_tie replaces,
    // or a row's output would depend on the rows beside it
    asm("add.u16x2 %0, %0, %1;" : "+r"(x) : "r"(0x80108010u));
    asm("min.u16x2 %0, %0, %1;" : "+r"(m) : "r"(x));
    return m;
}
__device__ __forceinline__ bool tie_found(uint32_t m) { return (m & 0xffffu) < 32u || (m >> 16) < 32u; }
__device__ __forceinline__ float at_tie(float g, float h)
{
    if (((__float_as_uint(g) + 0x8010u) & 0xffffu) >= 32u || fabsf(g) < 0.015625f) return g;
    return h * (1.0f + erff(2.0f * h * 0.70710678118654752f));
}

// gelu of 16 columns to be rounded to BF16: v holds the accumulators, half() gives the halved
// pre-activations from them, reload() the accumulators again (every lane of the warp calls it).
template <typename Half, typename Reload>
__device__ __forceinline__ void gelu16(float (&v)[16], Half &&half, Reload &&reload)
{
    uint32_t m = 0xffffffffu;
#pragma unroll
    for (int k = 0; k < 16; k += 2) {
        float h0, h1;
        upk(half(k, v[k], v[k + 1]), h0, h1);
        upk(gelu_pair(h0, h1), v[k], v[k + 1]);
        m = tie_key(m, v[k], v[k + 1]);
    }
    if (__any_sync(0xffffffffu, tie_found(m))) {
        float a[16];
        reload(a);
#pragma unroll
        for (int k = 0; k < 16; k += 2) {
            float h0, h1;
            upk(half(k, a[k], a[k + 1]), h0, h1);
            v[k] = at_tie(v[k], h0);
            v[k + 1] = at_tie(v[k + 1], h1);
        }
    }
}

// gelu and its derivative Phi(z) + z phi(z) of a pair z = 2 h.
__device__ __forceinline__ void gelu_grad_pair(float h0, float h1, f2 &g, f2 &d)
{
    const f2 s = pk(fmaxf(-fabsf(h0), -3.0f), fmaxf(-fabsf(h1), -3.0f));
    const f2 e = erfc_pair(s);
    g = fma2(s, e, pk(h0 + fabsf(h0), h1 + fabsf(h1)));
    // Phi = 1/2 + copysign((1 - erfc)/2, z); 1 - erfc/2 and erfc/2 taken directly
    float e0, e1;
    upk(mul2(e, pk(0.5f, 0.5f)), e0, e1);
    const float p0 = h0 >= 0.0f ? 1.0f - e0 : e0, p1 = h1 >= 0.0f ? 1.0f - e1 : e1;
    // phi(z) = exp(-z^2/2) / sqrt(2 pi); z phi = h 2 phi, -z^2/2 = -2 h^2
    const f2 h = pk(h0, h1);
    float x0, x1;
    upk(mul2(mul2(h, pk(-2.885390082f, -2.885390082f)), h), x0, x1);
    d = fma2(mul2(h, pk(0.79788456080f, 0.79788456080f)), pk(ex2(x0), ex2(x1)), pk(p0, p1));
}

}  // namespace gelu
}  // namespace sph

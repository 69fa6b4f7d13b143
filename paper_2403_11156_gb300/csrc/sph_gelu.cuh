// sph_gelu.cuh -- the network's exact GELU, z Phi(z), and its derivative.
//
//   gelu(z) = max(z, 0) - |z|/2 erfc(|z|/sqrt 2),   erfc(t/sqrt 2) = 2^Q(t),
//
// with Q a degree-9 polynomial without constant term fitted to log2 erfc(t/sqrt 2) on
// [0, 6] (minimax of the error times erfc, by iteratively reweighted least squares against
// 40-digit values).  No branch and one ex2 in place of erff's two polynomial branches and its exp: 8
// instructions an evaluation in the pairwise form below, about 28 before.  Error against
// 64-bit values over [-9, 9]: at most 2.4e-7 and 5.0e-8 rms, where 0.5 z (1 + erff(z/sqrt 2))
// has 4.5e-7 and 6.4e-8.  Beyond |z| = 6 erfc is held at its value there (2e-9).  NaN stays
// NaN, +inf gives +inf and -inf gives NaN, as the product form does.
#pragma once

#include <cuda_runtime.h>

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

// reg_dft.cuh -- DFTs of 3, 4, 5, 8, 12, 16 and 20 complex values held in one
// thread's registers, natural order in and out, for the one-CTA transform of
// conv_fft.cu.
//
// A complex value is one 64-bit register pair, so its sums and differences are
// single packed instructions (__fadd2_rn, __ffma2_rn: two float32 results, each
// rounded as the scalar operation rounds it).  Steps with a constant or a factor
// of i stay scalar FMAs: packed, they would need the constant in a register
// pair of its own and the halves swapped.
//
// 12 = 3 x 4 and 20 = 4 x 5 take the prime-factor maps (Good 1958): input
// n = (B a + A b) mod AB, output k from its residues, no twiddles between the
// two levels.  16 is two radix-4 levels with the eight distinct twiddles of
// W_16; 8 is a radix-2 level over two radix-4 ones.
// INV: exponent +2 pi i / N instead of -2 pi i / N.
#pragma once

#include <cuda_runtime.h>

__device__ __forceinline__ float2 c2(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ float2 c_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 c_sub(float2 a, float2 b) { return __ffma2_rn(b, c2(-1.0f, -1.0f), a); }
// a + s b for a real s
__device__ __forceinline__ float2 c_fma(float s, float2 b, float2 a) { return c2(fmaf(s, b.x, a.x), fmaf(s, b.y, a.y)); }
// a + s (-i b) forward, a + s (+i b) inverse, for a real s
template <bool INV>
__device__ __forceinline__ float2 c_addi(float s, float2 b, float2 a)
{
    return INV ? c2(fmaf(-s, b.y, a.x), fmaf(s, b.x, a.y)) : c2(fmaf(s, b.y, a.x), fmaf(-s, b.x, a.y));
}
__device__ __forceinline__ float2 c_mul(float2 a, float2 w)
{
    return c2(fmaf(a.x, w.x, -a.y * w.y), fmaf(a.x, w.y, a.y * w.x));
}
// a conj(w)
__device__ __forceinline__ float2 c_mulc(float2 a, float2 w)
{
    return c2(fmaf(a.x, w.x, a.y * w.y), fmaf(a.y, w.x, -a.x * w.y));
}

template <bool INV>
__device__ __forceinline__ void rdft3(float2& x0, float2& x1, float2& x2)
{
    const float2 t = c_add(x1, x2), d = c_sub(x1, x2);
    const float2 m = c_fma(-0.5f, t, x0);
    x0 = c_add(x0, t);
    x1 = c_addi<INV>(0.86602540378443865f, d, m);
    x2 = c_addi<INV>(-0.86602540378443865f, d, m);
}

template <bool INV>
__device__ __forceinline__ void rdft4(float2& x0, float2& x1, float2& x2, float2& x3)
{
    const float2 a = c_add(x0, x2), b = c_sub(x0, x2), c = c_add(x1, x3), d = c_sub(x1, x3);
    x0 = c_add(a, c);
    x2 = c_sub(a, c);
    x1 = c_addi<INV>(1.0f, d, b);
    x3 = c_addi<INV>(-1.0f, d, b);
}

template <bool INV>
__device__ __forceinline__ void rdft5(float2& x0, float2& x1, float2& x2, float2& x3, float2& x4)
{
    constexpr float C1 = 0.30901699437494742f, C2 = -0.80901699437494742f;  // cos 2 pi / 5, cos 4 pi / 5
    constexpr float S1 = 0.95105651629515357f, S2 = 0.58778525229247313f;   // sin of the same
    const float2 t1 = c_add(x1, x4), t2 = c_add(x2, x3), d1 = c_sub(x1, x4), d2 = c_sub(x2, x3);
    const float2 a1 = c_fma(C2, t2, c_fma(C1, t1, x0)), a2 = c_fma(C1, t2, c_fma(C2, t1, x0));
    x0 = c_add(x0, c_add(t1, t2));
    x1 = c_addi<INV>(S2, d2, c_addi<INV>(S1, d1, a1));
    x4 = c_addi<INV>(-S2, d2, c_addi<INV>(-S1, d1, a1));
    x2 = c_addi<INV>(-S1, d2, c_addi<INV>(S2, d1, a2));
    x3 = c_addi<INV>(S1, d2, c_addi<INV>(-S2, d1, a2));
}

template <bool INV>
__device__ __forceinline__ void rdft8(float2 (&x)[8])
{
    constexpr float R = 0.70710678118654752f;
    rdft4<INV>(x[0], x[2], x[4], x[6]);
    rdft4<INV>(x[1], x[3], x[5], x[7]);
    // odd outputs times W_8^k: k = 1 -> R (1 - i), 2 -> -i, 3 -> -R (1 + i) (forward)
    const float2 e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    const float2 o0 = x[1], o2 = x[5];
    const float2 o1 = c_addi<INV>(1.0f, x[3], x[3]);   // x (1 - i) forward
    const float2 o3 = c_addi<INV>(-1.0f, x[7], x[7]);  // x (1 + i) forward
    x[0] = c_add(e0, o0);
    x[4] = c_sub(e0, o0);
    x[1] = c_fma(R, o1, e1);
    x[5] = c_fma(-R, o1, e1);
    x[2] = c_addi<INV>(1.0f, o2, e2);
    x[6] = c_addi<INV>(-1.0f, o2, e2);
    x[3] = c_fma(-R, o3, e3);
    x[7] = c_fma(R, o3, e3);
}

// x W_16^E (forward), x conj(W_16^E) (inverse)
template <int E, bool INV>
__device__ __forceinline__ float2 w16(float2 x)
{
    constexpr float C[10] = {1.0f, 0.92387953251128676f, 0.70710678118654752f, 0.38268343236508977f, 0.0f,
                             -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128676f, -1.0f,
                             -0.92387953251128676f};
    constexpr float S[10] = {0.0f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128676f, 1.0f,
                             0.92387953251128676f, 0.70710678118654752f, 0.38268343236508977f, 0.0f,
                             -0.38268343236508977f};
    if (E == 0) return x;
    return INV ? c_mul(x, c2(C[E], S[E])) : c_mul(x, c2(C[E], -S[E]));
}

template <int M, bool INV>
__device__ __forceinline__ void rdft(float2 (&x)[M])
{
    float2 y[M];
    if constexpr (M == 12) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            y[b] = x[(3 * b) % 12], y[4 + b] = x[(4 + 3 * b) % 12], y[8 + b] = x[(8 + 3 * b) % 12];
            rdft3<INV>(y[b], y[4 + b], y[8 + b]);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            rdft4<INV>(y[4 * a], y[4 * a + 1], y[4 * a + 2], y[4 * a + 3]);
#pragma unroll
            for (int b = 0; b < 4; ++b) x[(4 * a + 9 * b) % 12] = y[4 * a + b];
        }
    } else if constexpr (M == 20) {
#pragma unroll
        for (int b = 0; b < 5; ++b) {
#pragma unroll
            for (int a = 0; a < 4; ++a) y[5 * a + b] = x[(5 * a + 4 * b) % 20];
            rdft4<INV>(y[b], y[5 + b], y[10 + b], y[15 + b]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            rdft5<INV>(y[5 * a], y[5 * a + 1], y[5 * a + 2], y[5 * a + 3], y[5 * a + 4]);
#pragma unroll
            for (int b = 0; b < 5; ++b) x[(5 * a + 16 * b) % 20] = y[5 * a + b];
        }
    } else {
        static_assert(M == 16, "12, 16 or 20 points");
#pragma unroll
        for (int a = 0; a < 4; ++a) rdft4<INV>(x[a], x[a + 4], x[a + 8], x[a + 12]);
        // x[a + 4 k] is output k of sub-transform a
        y[5] = w16<1, INV>(x[5]), y[9] = w16<2, INV>(x[9]), y[13] = w16<3, INV>(x[13]);
        y[6] = w16<2, INV>(x[6]), y[10] = w16<4, INV>(x[10]), y[14] = w16<6, INV>(x[14]);
        y[7] = w16<3, INV>(x[7]), y[11] = w16<6, INV>(x[11]), y[15] = w16<9, INV>(x[15]);
        y[0] = x[0], y[1] = x[1], y[2] = x[2], y[3] = x[3];
        y[4] = x[4], y[8] = x[8], y[12] = x[12];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            rdft4<INV>(y[4 * k], y[4 * k + 1], y[4 * k + 2], y[4 * k + 3]);
#pragma unroll
            for (int a = 0; a < 4; ++a) x[k + 4 * a] = y[4 * k + a];
        }
    }
}

// cnn.cu -- the learned initial guess: a small convolutional network that maps
// a 64x64 stamp to the eight regression targets of a single Sersic component,
// its training data drawn on the device, the moments-based default guess, and
// the choice between the two starts.
//
// Network (NCHW, one 64x64 input channel, zero padding 1, stride 2, ReLU after
// every layer but the last):
//   conv 3x3 1->32 (64->32), 32->64 (32->16), 64->64 (16->8), 64->128 (8->4),
//   fc 2048->32, fc 32->8.
// Weights and activations are bf16, every accumulation float32.  The master
// parameters are float32, packed layer by layer as weights [out][in][ky][kx]
// (fc: [out][in]) then biases [out] -- 195432 in all.  Two bf16 copies of the
// convolution weights are kept: [in][tap][out] for the forward pass (eight
// consecutive output channels per 16-byte load; the first layer's SIMT loop and
// the tensor-core input gradients read it) and [out][tap][in] (the tensor-core
// forward's B operand).  The convolution layers' activations and gradients are
// channels-last except conv4's output, which is stored in the [c][y][x] order
// fc1 flattens.  Convolutions 2-4 run on the tensor cores in both directions
// (cnn_tc.cu, cnn_bwd_tc.cu); this file holds the first convolution, the fully
// connected layers, the loss and Adam.  Every reduction runs in a fixed order,
// so a training run is reproducible bit for bit.
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "bn.cuh"
#include "cnn.cuh"
#include "gf_internal.cuh"

namespace {

struct ConvL {
    int cin, cout, hin, hout;
    int woff, boff;  // offsets in the master parameter array
};

#define CONV_TABLE                                                                              \
    {                                                                                           \
        {1, 32, 64, 32, 0, 288}, {32, 64, 32, 16, 320, 18752}, {64, 64, 16, 8, 18816, 55680}, \
            {64, 128, 8, 4, 55744, 129472}                                                      \
    }
constexpr ConvL CONV[4] = CONV_TABLE;
__constant__ ConvL c_conv[4] = CONV_TABLE;

constexpr int FC1_W = 129600, FC1_B = 195136, FC2_W = 195168, FC2_B = 195424;
constexpr int NPARAM = CNN_NPARAM;
constexpr int CONV_W_END = 129600;  // the conv weights and biases occupy [0, CONV_W_END)
constexpr int SIDE = CNN_SIDE, NPIX = SIDE * SIDE, NOUT = CNN_NOUT;

__device__ __forceinline__ void unpack8(const uint4 u, float* f)
{
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 t = __bfloat1622float2(h[i]);
        f[2 * i] = t.x;
        f[2 * i + 1] = t.y;
    }
}

inline int blocks(long long n, int t) { return (int)((n + t - 1) / t); }

// ---------------------------------------------------------------- forward
// fc1: thread = (NB samples, o); input the flattened conv4 output (bf16), output
// float32 after ReLU.  A lane's weights are a row of their own (32 sectors a load),
// which is what bounds it, so NB samples share them; four loads stay in flight.
// 8,192 stamps (NB 4): 257 us -> 101.  Below 2,048 samples a sample a thread: four would
// leave most SMs without a block.
template <int NB>
__global__ void k_fc1_fwd(const __nv_bfloat16* __restrict__ a3, const __nv_bfloat16* __restrict__ w,
                          const float* __restrict__ master, float* __restrict__ h, int B)
{
    const int item = blockIdx.x * blockDim.x + threadIdx.x;
    const int b0 = (item >> 5) * NB, o = item & 31;
    if (b0 >= B) return;
    const __nv_bfloat16* xr[NB];
    float acc[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
        xr[q] = a3 + (long long)min(b0 + q, B - 1) * 2048;
        acc[q] = master[FC1_B + o];
    }
    const __nv_bfloat16* wr = w + FC1_W + o * 2048;
#pragma unroll 4
    for (int i = 0; i < 2048; i += 8) {
        float wv[8];
        unpack8(*reinterpret_cast<const uint4*>(wr + i), wv);
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            float xv[8];
            unpack8(*reinterpret_cast<const uint4*>(xr[q] + i), xv);
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[q] = fmaf(xv[j], wv[j], acc[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < NB; ++q)
        if (b0 + q < B) h[(b0 + q) * 32 + o] = fmaxf(acc[q], 0.0f);
}

// fc2: thread = (b, j); linear output
__global__ void k_fc2_fwd(const float* __restrict__ h, const __nv_bfloat16* __restrict__ w,
                          const float* __restrict__ master, float* __restrict__ y, int B)
{
    const int item = blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= B * NOUT) return;
    const int b = item / NOUT, j = item - b * NOUT;
    float acc = master[FC2_B + j];
    for (int o = 0; o < 32; ++o)
        acc = fmaf(__bfloat162float(w[FC2_W + j * 32 + o]), h[b * 32 + o], acc);
    y[item] = acc;
}

// ------------------------------------------------------------------ loss
// loss = mean (y - t)^2 over B x 8 (one block, fixed-order tree); gy = dloss/dy
__global__ void k_mse(const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ gy,
                      float* __restrict__ loss, int B)
{
    __shared__ float part[256];
    const int n = B * NOUT;
    const float scale = 1.0f / (float)n;
    float s = 0.0f;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float e = y[i] - t[i];
        gy[i] = 2.0f * e * scale;
        s = fmaf(e, e, s);
    }
    part[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = part[0] * scale;
}

// -------------------------------------------------------------- backward
// fc2: weight/bias gradients (thread per (j, o) / j, summed over the batch)
__global__ void k_fc2_bwd_w(const float* __restrict__ gy, const float* __restrict__ h,
                            float* __restrict__ grad, int B)
{
    const int item = blockIdx.x * blockDim.x + threadIdx.x;
    if (item < NOUT * 32) {
        const int j = item / 32, o = item - j * 32;
        float s = 0.0f;
#pragma unroll 16  // (the loads of 16 samples in flight; the sum stays in order)
        for (int b = 0; b < B; ++b) s = fmaf(gy[b * NOUT + j], h[b * 32 + o], s);
        grad[FC2_W + item] = s;
    } else if (item < NOUT * 32 + NOUT) {
        const int j = item - NOUT * 32;
        float s = 0.0f;
#pragma unroll 16
        for (int b = 0; b < B; ++b) s += gy[b * NOUT + j];
        grad[FC2_B + j] = s;
    }
}

// gradient at fc1's pre-activation
__global__ void k_fc2_bwd_x(const float* __restrict__ gy, const float* __restrict__ h,
                            const __nv_bfloat16* __restrict__ w, float* __restrict__ gh, int B)
{
    const int item = blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= B * 32) return;
    const int b = item / 32, o = item - b * 32;
    float s = 0.0f;
    for (int j = 0; j < NOUT; ++j) s = fmaf(__bfloat162float(w[FC2_W + j * 32 + o]), gy[b * NOUT + j], s);
    gh[item] = h[item] > 0.0f ? s : 0.0f;
}

// fc1 weight (thread per (o, i)) and bias gradients
__global__ void k_fc1_bwd_w(const float* __restrict__ gh, const __nv_bfloat16* __restrict__ a3,
                            float* __restrict__ grad, int B)
{
    const int item = blockIdx.x * blockDim.x + threadIdx.x;
    if (item < 32 * 2048) {
        const int o = item / 2048, i = item - o * 2048;
        float s = 0.0f;
#pragma unroll 16
        for (int b = 0; b < B; ++b) s = fmaf(gh[b * 32 + o], __bfloat162float(a3[(long long)b * 2048 + i]), s);
        grad[FC1_W + item] = s;
    } else if (item < 32 * 2048 + 32) {
        const int o = item - 32 * 2048;
        float s = 0.0f;
#pragma unroll 16
        for (int b = 0; b < B; ++b) s += gh[b * 32 + o];
        grad[FC1_B + o] = s;
    }
}

// gradient at conv4's pre-activation (through its ReLU), written channels-last
// (b, pixel, channel) for the tensor-core backward; the flattened input index i
// of fc1 is channel * 16 + pixel (conv4's NCHW output)
__global__ void k_fc1_bwd_x(const float* __restrict__ gh, const __nv_bfloat16* __restrict__ a3,
                            const __nv_bfloat16* __restrict__ w, float* __restrict__ g3, int B)
{
    const long long item = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= (long long)B * 2048) return;
    const int b = (int)(item / 2048), i = (int)(item - (long long)b * 2048);
    float s = 0.0f;
    for (int o = 0; o < 32; ++o) s = fmaf(__bfloat162float(w[FC1_W + o * 2048 + i]), gh[b * 32 + o], s);
    const int c = i >> 4, pix = i & 15;
    g3[(long long)b * 2048 + pix * 128 + c] = __bfloat162float(a3[item]) > 0.0f ? s : 0.0f;
}

// Weight gradients of the first convolution (one input channel, nine taps per
// output channel: too narrow for the tensor cores), first stage: block =
// (8 output channels, chunk of the batch); threads stride over (b, oy, ox),
// keeping for each channel the nine tap sums and the bias sum; a fixed tree merges
// the threads.  gout is channels-last (b, oy, ox, co), so 8 channels are the 32
// bytes that a pixel's read fetches in any case, and the nine inputs are read once
// for the 8 (a block per channel: 174 us on 512 stamps, 74 now).
constexpr int WG_THREADS = 256;
constexpr int WG_CO = 8;  // channels a block

__global__ void __launch_bounds__(WG_THREADS) k_conv_bwd_w(const float* __restrict__ gout,
                                                            const __nv_bfloat16* __restrict__ xin,
                                                            float* __restrict__ part, int B, int hin,
                                                            int cout, int hout, int nchunk)
{
    __shared__ float red[10][WG_THREADS];
    const int co0 = blockIdx.x * WG_CO, chunk = blockIdx.y;
    const int npix = hout * hout, lho = __ffs(hout) - 1;  // (a power of two)
    const long long total = (long long)B * npix;
    const long long per = (total + nchunk - 1) / nchunk;
    const long long i0 = chunk * per, i1 = min(total, i0 + per);
    float s[WG_CO][10];
#pragma unroll
    for (int j = 0; j < WG_CO; ++j)
#pragma unroll
        for (int k = 0; k < 10; ++k) s[j][k] = 0.0f;
    for (long long it = i0 + threadIdx.x; it < i1; it += WG_THREADS) {
        const int b = (int)(it >> (2 * lho)), pix = (int)it & (npix - 1);
        const int oy = pix >> lho, ox = pix & (hout - 1);
        const float4* gp = reinterpret_cast<const float4*>(gout + it * cout + co0);
        const float4 g0 = gp[0], g1 = gp[1];
        const float g[WG_CO] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
        const __nv_bfloat16* xb = xin + (long long)b * hin * hin;
        float x[9];
        bool in[9];  // taps inside the image
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int iy = 2 * oy - 1 + t / 3, ix = 2 * ox - 1 + t % 3;
            in[t] = iy >= 0 && iy < hin && ix >= 0 && ix < hin;
            x[t] = in[t] ? __bfloat162float(xb[iy * hin + ix]) : 0.0f;
        }
#pragma unroll
        for (int j = 0; j < WG_CO; ++j) {
            if (g[j] == 0.0f) continue;  // (also where the input is not finite)
            s[j][9] += g[j];
#pragma unroll
            for (int t = 0; t < 9; ++t)
                if (in[t]) s[j][t] = fmaf(g[j], x[t], s[j][t]);
        }
    }
#pragma unroll
    for (int j = 0; j < WG_CO; ++j) {
        __syncthreads();  // (the sums of the channel before are out)
#pragma unroll
        for (int k = 0; k < 10; ++k) red[k][threadIdx.x] = s[j][k];
        __syncthreads();
        for (int w = WG_THREADS / 2; w > 0; w >>= 1) {
            if (threadIdx.x < w)
#pragma unroll
                for (int k = 0; k < 10; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
            __syncthreads();
        }
        // part layout: [chunk][co][10]
        if (threadIdx.x < 10) part[((long long)chunk * cout + co0 + j) * 10 + threadIdx.x] = red[threadIdx.x][0];
    }
}

// second stage: the chunks summed in order into the packed master layout
__global__ void k_conv_bwd_w_sum(const float* __restrict__ part, float* __restrict__ grad, int cin,
                                 int cout, int nchunk, int woff, int boff)
{
    const int item = blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= cout * cin * 10) return;
    float s = 0.0f;
    for (int c = 0; c < nchunk; ++c) s += part[(long long)c * cout * cin * 10 + item];
    const int k = item % 10, pair = item / 10, ci = pair % cin, co = pair / cin;
    if (k < 9)
        grad[woff + (co * cin + ci) * 9 + k] = s;
    else if (ci == 0)
        grad[boff + co] = s;
}

// ------------------------------------------------------------ optimiser
// Adam (Kingma & Ba 2015) on the float32 masters; c1, c2 = bias corrections
__global__ void k_adam(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, int n, float lr, float b1, float b2, float eps,
                       float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// bf16 copies of the masters: the packed layout, plus the two transposed
// layouts of the convolution weights
__global__ void k_cast(const float* __restrict__ w, __nv_bfloat16* __restrict__ wp,
                       __nv_bfloat16* __restrict__ wf, __nv_bfloat16* __restrict__ wb)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NPARAM) return;
    const __nv_bfloat16 h = __float2bfloat16_rn(w[i]);
    wp[i] = h;
    if (i >= CONV_W_END) return;
    for (int l = 0; l < 4; ++l) {
        const ConvL L = c_conv[l];
        if (i < L.woff || i >= L.boff) continue;
        const int r = i - L.woff, co = r / (L.cin * 9), ci = (r / 9) % L.cin, tap = r % 9;
        wf[L.woff + (ci * 9 + tap) * L.cout + co] = h;  // [in][tap][out]
        wb[L.woff + (co * 9 + tap) * L.cin + ci] = h;   // [out][tap][in]
    }
}

__global__ void k_to_bf16(const float* __restrict__ x, __nv_bfloat16* __restrict__ y, long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = __float2bfloat16_rn(x[i]);
}

// ---------------------------------------------------------------- Philox
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC 2011): ten rounds, each
// multiplying words 0 and 2 by the round constants 0xD2511F53 and 0xCD9E8D57,
// swapping in the high halves xored with the other words and the key, and
// bumping the key by the Weyl constants 0x9E3779B9, 0xBB67AE85.
__device__ __forceinline__ uint4 philox(uint4 ctr, uint2 key)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned hi0 = __umulhi(0xD2511F53u, ctr.x), lo0 = 0xD2511F53u * ctr.x;
        const unsigned hi1 = __umulhi(0xCD9E8D57u, ctr.z), lo1 = 0xCD9E8D57u * ctr.z;
        ctr = make_uint4(hi1 ^ ctr.y ^ key.x, lo1, hi0 ^ ctr.w ^ key.y, lo0);
        key.x += 0x9E3779B9u;
        key.y += 0xBB67AE85u;
    }
    return ctr;
}

__device__ __forceinline__ uint2 key_of(unsigned long long seed)
{
    return make_uint2((unsigned)seed, (unsigned)(seed >> 32));
}

// a uniform in (0, 1) from one 32-bit word
__device__ __forceinline__ double unit(unsigned r) { return ((double)r + 0.5) * (1.0 / 4294967296.0); }

// one standard normal from counter (n, stream) by the Box-Muller transform
__device__ __forceinline__ float normal1(unsigned long long n, unsigned stream, uint2 key)
{
    const uint4 r = philox(make_uint4((unsigned)n, (unsigned)(n >> 32), stream, 0u), key);
    const float u1 = (float)unit(r.x), u2 = (float)unit(r.y);
    return sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
}

__global__ void k_philox(const unsigned* __restrict__ in, unsigned* __restrict__ out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const unsigned* a = in + 6 * i;
    const uint4 r = philox(make_uint4(a[0], a[1], a[2], a[3]), make_uint2(a[4], a[5]));
    out[4 * i] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
}

// sigma^2 = sigma_read^2 + max(m, 0) / gain; d = m + sigma z
__global__ void k_noise(const float* __restrict__ m, long long n, unsigned long long seed, float sread,
                        float gain, float* __restrict__ d, float* __restrict__ sig)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float mi = m[i];
    const float s = sqrtf(sread * sread + fmaxf(mi, 0.0f) / gain);
    d[i] = mi + s * normal1((unsigned long long)i, 0u, key_of(seed));
    sig[i] = s;
}

// He-normal initial weights N(0, 2 / fan_in), biases 0
__global__ void k_init(float* __restrict__ w, unsigned long long seed)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NPARAM) return;
    int fan = 0;
    for (int l = 0; l < 4; ++l)
        if (i >= c_conv[l].woff && i < c_conv[l].boff) fan = c_conv[l].cin * 9;
    if (i >= FC1_W && i < FC1_B) fan = 2048;
    if (i >= FC2_W && i < FC2_B) fan = 32;
    w[i] = fan ? normal1((unsigned long long)i, 1u, key_of(seed)) * sqrtf(2.0f / (float)fan) : 0.0f;
}

// --------------------------------------------------- b_n and Sersic flux
// Regularised lower incomplete gamma by its power series
//   P(a, x) = x^a e^{-x} / Gamma(a+1) * sum_k x^k / ((a+1)...(a+k)),
// for 0 < x < a <= 20: the terms fall, and the 64th is below 1e-17 of the sum.
// The sum 1 + x/(a+1) (1 + x/(a+2) (1 + ...)) is carried from its innermost
// bracket outwards as a quotient p / q, two multiplications a term and one
// division in all (a division a term is most of the chain otherwise); q stays
// below 84! / 20! < 1e109.
__device__ double gamma_p(double a, double x, double lg1)
{
    if (x <= 0.0) return 0.0;
    double p = 1.0, q = 1.0;
#pragma unroll 8
    for (int k = 64; k >= 1; --k) {
        q *= a + k;
        p = fma(x, p, q);
    }
    return exp(a * log(x) - x - lg1) * (p / q);
}

// b_n: root of P(2n, b) = 1/2 by Halley steps inside a bisection bracket
// (0, 2n), started from the asymptotic series of Ciotti & Bertin (1999).  Each
// evaluation of P is a long chain of FP64 divisions, so the cubic step pays:
// P' is the Gamma density and P'' / P' = (a - 1) / b - 1, both free once P is
// known.  A step below 1e-6 b leaves an error of order 1e-18 b, so the loop ends
// with it (one to three evaluations of P over n in [0.2, 10]).
__device__ double bn_of(double n)
{
    const double a = 2.0 * n;
    double lo = 0.0, hi = a;
    double b = a - 1.0 / 3.0 + 4.0 / (405.0 * n) + 46.0 / (25515.0 * n * n);
    if (!(b > lo && b < hi)) b = 0.5 * a;
    const double lg1 = lgamma(a + 1.0), lga = lg1 - log(a);
    for (int it = 0; it < 200; ++it) {
        const double f = gamma_p(a, b, lg1) - 0.5;
        if (f == 0.0) break;
        if (f < 0.0)
            lo = b;
        else
            hi = b;
        const double u = f / exp((a - 1.0) * log(b) - b - lga);  // f / f'
        double nb = b - u / (1.0 - 0.5 * u * ((a - 1.0) / b - 1.0));
        // (at the root the step vanishes and nb is b, an end of the bracket: that
        // is the end too, not a reason to bisect)
        const bool done = fabs(u) <= 1e-6 * b;
        if (!done && !(nb > lo && nb < hi)) nb = 0.5 * (lo + hi);
        b = nb;
        if (done || hi - lo <= 1e-15 * b) break;
    }
    return b;
}

// the n-dependent factor e^{b} Gamma(2n) / b^{2n} of the closed-form flux
__device__ double sersic_flux_factor(double n)
{
    const double b = bn_of(n);
    return exp(b + lgamma(2.0 * n) - 2.0 * n * log(b));
}

// closed-form total flux of an elliptical Sersic component:
// 2 pi q I_e r_e^2 n e^{b} Gamma(2n) / b^{2n}, given its n-dependent factor e
__device__ double sersic_flux_e(double ie, double re, double n, double q, double e)
{
    return 2.0 * M_PI * q * ie * re * re * n * e;
}

__device__ double sersic_flux(double ie, double re, double n, double q)
{
    return sersic_flux_e(ie, re, n, q, sersic_flux_factor(n));
}

// the factor at n = 2 (the default guess's index), b_2 = 3.6720607488508961
constexpr double kFluxFactorN2 = 1.2979786274281866;

// ------------------------------------------------ network input scaling
template <class T>
__device__ void bitonic_sort(T* v, int n)  // n a power of two
{
    for (int k = 2; k <= n; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = threadIdx.x; t < n / 2; t += blockDim.x) {
                const int i = 2 * t - (t & (j - 1));
                const int p = i + j;
                const bool up = (i & k) == 0;
                const T a = v[i], b = v[p];
                if ((a > b) == up) {
                    v[i] = b;
                    v[p] = a;
                }
            }
            __syncthreads();
        }
}

// pixel k of the outer ring: top row, bottom row, then the left and right
// columns without their corners
__device__ __forceinline__ void ring_ij(int k, int H, int W, int* i, int* j)
{
    if (k < W) {
        *i = 0;
        *j = k;
    } else if (k < 2 * W) {
        *i = H - 1;
        *j = k - W;
    } else if (k < 2 * W + (H - 2)) {
        *i = k - 2 * W + 1;
        *j = 0;
    } else {
        *i = k - 2 * W - (H - 2) + 1;
        *j = W - 1;
    }
}

// block per stamp: a = median of sigma over the outer ring (252 pixels, mean
// of the two middle values), x = asinh(img / a)
__global__ void __launch_bounds__(256) k_cnn_input(const float* __restrict__ img,
                                                    const float* __restrict__ sig,
                                                    float* __restrict__ x)
{
    __shared__ float v[256];
    const long long base = (long long)blockIdx.x * NPIX;
    constexpr int NR = 4 * SIDE - 4;
    if (threadIdx.x < NR) {
        int i, j;
        ring_ij(threadIdx.x, SIDE, SIDE, &i, &j);
        v[threadIdx.x] = sig[base + i * SIDE + j];
    } else {
        v[threadIdx.x] = INFINITY;
    }
    __syncthreads();
    bitonic_sort(v, 256);
    float a = 0.5f * (v[NR / 2 - 1] + v[NR / 2]);
    if (!(a > 0.0f)) a = 1.0f;
    for (int k = threadIdx.x; k < NPIX; k += blockDim.x) x[base + k] = asinhf(img[base + k] / a);
}

// ------------------------------------------------------ training stamps
// Stamp b of the training batch keyed by `seed`: the Sersic + sky parameters
// (9 slots) drawn from the training prior, and the Moffat PSF (beta 3, FWHM
// ~ U[2, 5]) on a psf_size^2 grid, normalised in float64.  Prior: centre
// (31.5, 31.5) + U[-1, 1] each; n ~ U[0.5, 6]; r_e log-uniform [2, 40];
// q ~ U[0.2, 1]; pa ~ U[0, 180); flux log-uniform [1e2, 1e5]; sky 0.05.
__global__ void __launch_bounds__(256) k_train_sample(unsigned long long seed, double* __restrict__ params,
                                                       float* __restrict__ psf, int psf_size)
{
    __shared__ double red[256];
    __shared__ double s_alpha;
    const int b = blockIdx.x;
    if (threadIdx.x < 32) {
        // warp 0: every lane draws the same values; the warp solves for b_n
        const uint2 key = key_of(seed);
        const uint4 r0 = philox(make_uint4((unsigned)b, 0u, 2u, 0u), key);
        const uint4 r1 = philox(make_uint4((unsigned)b, 1u, 2u, 0u), key);
        const double c = 0.5 * (SIDE - 1);
        const double n = 0.5 + 5.5 * unit(r0.z);
        const double bn = sersic_bn_warp(n, -1.0);
        const double re = exp(log(2.0) + (log(40.0) - log(2.0)) * unit(r0.w));
        const double q = 0.2 + 0.8 * unit(r1.x);
        const double pa = 180.0 * unit(r1.y);
        const double F = exp(log(1e2) + (log(1e5) - log(1e2)) * unit(r1.z));
        const double fwhm = 2.0 + 3.0 * unit(r1.w);
        double* p = params + 9 * (long long)b;
        if (threadIdx.x == 0) {
            p[0] = c - 1.0 + 2.0 * unit(r0.x);
            p[1] = c - 1.0 + 2.0 * unit(r0.y);
            p[2] = F / sersic_flux_e(1.0, re, n, q, exp(bn + lgamma(2.0 * n) - 2.0 * n * log(bn)));
            p[3] = re;
            p[4] = n;
            p[5] = q;
            p[6] = pa;
            p[7] = 0.0;
            p[8] = 0.05;
            s_alpha = fwhm / (2.0 * sqrt(exp2(1.0 / 3.0) - 1.0));
        }
    }
    __syncthreads();
    const int c = psf_size / 2, np = psf_size * psf_size;
    const double ia2 = 1.0 / (s_alpha * s_alpha);
    double s = 0.0;
    for (int k = threadIdx.x; k < np; k += blockDim.x) {
        const int y = k / psf_size - c, x = k % psf_size - c;
        const double u = 1.0 + (double)(x * x + y * y) * ia2;
        s += 1.0 / (u * u * u);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    const double inv = 1.0 / red[0];
    for (int k = threadIdx.x; k < np; k += blockDim.x) {
        const int y = k / psf_size - c, x = k % psf_size - c;
        const double u = 1.0 + (double)(x * x + y * y) * ia2;
        psf[(long long)b * np + k] = (float)(inv / (u * u * u));
    }
}

// targets of the first Sersic component (slots 0..6 of a stamp's parameters)
// a warp per stamp (the warp solves for b_n), lane 0 writes the targets
__global__ void k_encode(const double* __restrict__ params, int nslots, int count, int H, int W,
                         float* __restrict__ t)
{
    const int b = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (b >= count) return;  // the whole warp
    const double* p = params + (long long)b * nslots;
    const double bn = sersic_bn_warp(p[4], -1.0);
    if ((threadIdx.x & 31) != 0) return;
    const double l10 = log(10.0);
    const double th = 2.0 * p[6] * M_PI / 180.0;
    float* o = t + (long long)b * NOUT;
    o[0] = (float)(p[0] - 0.5 * (W - 1));
    o[1] = (float)(p[1] - 0.5 * (H - 1));
    const double e = exp(bn + lgamma(2.0 * p[4]) - 2.0 * p[4] * log(bn));
    o[2] = (float)((log(sersic_flux_e(p[2], p[3], p[4], p[5], e)) - 3.5 * l10) / (1.5 * l10));
    o[3] = (float)((log(p[3]) - 0.5 * log(80.0)) / (0.5 * log(20.0)));
    o[4] = (float)((p[4] - 3.25) / 2.75);
    o[5] = (float)((p[5] - 0.6) / 0.4);
    o[6] = (float)cos(th);
    o[7] = (float)sin(th);
}

// inverse of k_encode: Sersic slots (c = 0) plus the sky slot copied from the
// default guess (and its centre, with GF_DECODE_MOMENT_CENTRE); I_e is NaN
// outside the closed-form flux domain
__global__ void k_decode(const float* __restrict__ y, const double* __restrict__ dflt, int count,
                         int H, int W, int flags, double* __restrict__ params)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= count) return;
    const float* t = y + (long long)b * NOUT;
    double* p = params + (long long)b * 9;
    const double l10 = log(10.0);
    const double F = exp(3.5 * l10 + 1.5 * l10 * t[2]);
    const double re = exp(0.5 * log(80.0) + 0.5 * log(20.0) * t[3]);
    const double n = 3.25 + 2.75 * t[4];
    const double q = 0.6 + 0.4 * t[5];
    double pa = 0.5 * atan2((double)t[7], (double)t[6]) * 180.0 / M_PI;
    if (pa < 0.0) pa += 180.0;
    p[0] = 0.5 * (W - 1) + t[0];
    p[1] = 0.5 * (H - 1) + t[1];
    p[2] = (n >= 0.2 && n <= 10.0 && q > 0.0 && q <= 1.0) ? F / sersic_flux(1.0, re, n, q) : NAN;
    p[3] = re;
    p[4] = n;
    p[5] = q;
    p[6] = pa;
    p[7] = 0.0;
    p[8] = dflt[(long long)b * 9 + 8];
    if (flags & GF_DECODE_MOMENT_CENTRE) {
        p[0] = dflt[(long long)b * 9];
        p[1] = dflt[(long long)b * 9 + 1];
    }
}

// ------------------------------------------------------- default guess
// Block per stamp of a batch.  Sky = median of the outer ring; centre = first
// moments of the sky-subtracted positive pixels; q and pa from the second
// moments; r_e = semi-major axis of the first elliptical aperture, in 0.25 px
// steps, holding half their summed flux (the enclosed flux only grows with the
// aperture's index); n = 2; I_e from the summed flux by the closed form.
//
// Every sum is float64 and the aperture test takes the decisions of a plain
// float64 evaluation without contracted multiply-adds.  What bounds the kernel
// is the FP64 pipe (two lanes per SM and clock: 16 cycles a warp instruction),
// so the split keeps as much as it can off it:
//   - the ring's median is selected on the float bit patterns;
//   - a lane owns a column while its warp walks the rows, so the moments need
//     per pixel the difference v and two or three accumulations, with the
//     column's factors applied once per column;
//   - a pixel's aperture index comes from a float32 radius; only pixels whose
//     radius lies within its error of an aperture take the float64 test;
//   - the half-light index is guessed from an integer histogram of the fluxes
//     over the aperture indices and proved by the float64 sums on both sides of
//     it (one pass instead of log2(4 max(H, W)) of them); where the proof fails
//     the index is found by bisection over the same sums.
// 8,192 stamps of 64x64: 7.0 ms -> 1.45 ms (the plain form of the same sums, one
// bisection pass per step and a float64 bitonic sort of the ring, before).
constexpr int DG_THREADS = 128, DG_WARPS = DG_THREADS / 32;
constexpr int DG_ROWS = 256;    // rows whose float64 offsets are tabulated
constexpr int DG_BINS = 1026;   // histogram bins: indices 0 .. 4 max(H, W) + 1

// N block-wide float64 sums, in every thread (two barriers)
template <int N>
__device__ __forceinline__ void block_sums(double (&v)[N], double (*red)[DG_WARPS])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < N; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
        if (lane == 0) red[q][warp] = v[q];
    }
    __syncthreads();
    if (threadIdx.x < N) {
        double t = red[threadIdx.x][0];
#pragma unroll
        for (int w = 1; w < DG_WARPS; ++w) t += red[threadIdx.x][w];
        red[threadIdx.x][0] = t;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = red[q][0];
    __syncthreads();
}

// float bit patterns as unsigned keys of the same order (and back)
__device__ __forceinline__ unsigned order_key(float f)
{
    const unsigned u = __float_as_uint(f);
    return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float order_value(unsigned k)
{
    return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu));
}

// (double)x off the FP64 pipe, which a conversion instruction would take: the
// exponent rebiased by integer operations; zeros, denormals, infinities and NaN
// are left to the instruction
__device__ __forceinline__ double widen(float x)
{
    const unsigned u = __float_as_uint(x);
    if ((((u >> 23) + 1u) & 0xfeu) == 0u) return (double)x;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// number of the n keys that are <= k (every thread)
__device__ __forceinline__ int count_le(const unsigned* key, int n, unsigned k)
{
    int c = 0;
    for (int t = 0; t < n; t += DG_THREADS)
        c += __syncthreads_count(t + (int)threadIdx.x < n && key[min(t + (int)threadIdx.x, n - 1)] <= k);
    return c;
}

// The stamp's geometry after the moments: what the aperture test needs
struct Ellipse {
    double x0, y0, cs, sn, q;
    float csf, snf, invqf;
};

// smallest aperture index k >= 1 with rr <= (0.25 k)^2 for the pixel's squared
// elliptical radius rr (dx = j - x0 and dy = i - y0 with their float values)
__device__ __forceinline__ int aperture_index(const Ellipse& e, int i, int j, float dx, float dy, int K)
{
    const float xp = fmaf(dx, e.csf, dy * e.snf);
    const float yp = fmaf(dy, e.csf, -dx * e.snf) * e.invqf;
    const float r4 = 4.0f * sqrtf(fmaf(xp, xp, yp * yp));
    // the float radius is good to a few units of 2^-24 (|dx| + |dy|) (1 + 1/q)
    const float tol = fmaf(4e-6f * (fabsf(dx) + fabsf(dy)), 1.0f + e.invqf, 1e-6f);
    const float near = rintf(r4);
    int k;
    if (fabsf(r4 - near) > tol) {
        k = r4 > (float)K ? K + 1 : (int)ceilf(r4);
    } else {
        const double ddx = j - e.x0, ddy = i - e.y0;
        const double xd = __dadd_rn(__dmul_rn(ddx, e.cs), __dmul_rn(ddy, e.sn));
        const double yd = __ddiv_rn(__dadd_rn(-__dmul_rn(ddx, e.sn), __dmul_rn(ddy, e.cs)), e.q);
        const double rr = __dadd_rn(__dmul_rn(xd, xd), __dmul_rn(yd, yd));
        auto in = [&](int m) {
            const double a = 0.25 * m;
            return rr <= __dmul_rn(a, a);
        };
        const double kd = ceil(4.0 * sqrt(rr));
        k = kd > (double)K ? K + 1 : (int)kd;
        while (k > 1 && in(k - 1)) --k;
        while (k <= K && !in(k)) ++k;
    }
    return max(k, 1);
}

// TAB: every stamp has at most DG_ROWS rows; CACHED: and at most cache_cap pixels
// (compile-time, since a select would evaluate the untabulated float64 forms too)
template <bool TAB, bool CACHED>
__global__ void __launch_bounds__(DG_THREADS) k_default_guess(const int* __restrict__ Hs,
                                                               const int* __restrict__ Ws,
                                                               const long long* __restrict__ off,
                                                               const float* __restrict__ img,
                                                               double* __restrict__ out, int nslots,
                                                               int ring_cap, int cache_cap)
{
    // dynamic shared memory: the ring's keys (ring_cap), then, for stamps of at
    // most cache_cap pixels, their v (0 where a pixel does not count) and their
    // aperture indices (0 there too)
    extern __shared__ __align__(16) unsigned ring[];
    __shared__ double red[3][DG_WARPS];
    __shared__ double dyt[DG_ROWS], dy2t[DG_ROWS];
    __shared__ float dyf[DG_ROWS];
    __shared__ unsigned hist[DG_BINS];
    __shared__ int s_k;
    __shared__ unsigned s_next;
    __shared__ Ellipse sc;
    __shared__ double s_pa;
    __shared__ float s_scale;
    const int b = blockIdx.x;
    const int H = Hs[b], W = Ws[b];
    const float* im = img + off[b];
    const int npx = H * W;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool line = H == 1 || W == 1;
    const int nr = line ? npx : 2 * W + 2 * (H - 2);
    for (int k = threadIdx.x; k < nr; k += DG_THREADS) {
        int i = 0, j = k;
        if (!line) ring_ij(k, H, W, &i, &j);
        ring[k] = order_key(im[i * W + j]);  // a single row or column is its own ring, in storage order
    }
    double* cv = reinterpret_cast<double*>(ring + ring_cap);
    unsigned short* idx = reinterpret_cast<unsigned short*>(cv + cache_cap);
    for (int i = threadIdx.x; i < (TAB ? H : 0); i += DG_THREADS) dyt[i] = (double)i;
    if (threadIdx.x == 0) s_next = 0xffffffffu;
    __syncthreads();
    // the ring's order statistic r1 (the lower middle one), bit by bit: the
    // largest prefix below which at most r1 keys lie; then the next one up
    const int r1 = (nr - 1) / 2;
    unsigned k1 = 0u;
    for (unsigned bit = 0x80000000u; bit != 0u; bit >>= 1) {
        const unsigned t = k1 | bit;
        if (count_le(ring, nr, t - 1u) <= r1) k1 = t;
    }
    double sky = (double)order_value(k1);
    if ((nr & 1) == 0) {
        if (count_le(ring, nr, k1) <= r1 + 1) {
            unsigned m = 0xffffffffu;
            for (int k = threadIdx.x; k < nr; k += DG_THREADS)
                if (ring[k] > k1) m = min(m, ring[k]);
            m = __reduce_min_sync(0xffffffffu, m);
            if (lane == 0) atomicMin(&s_next, m);
            __syncthreads();
            sky = 0.5 * (sky + (double)order_value(s_next));
        }
    }
    // v = pixel - sky counts where !(v <= 0): for a finite sky that is the
    // float test !(pixel <= sky rounded down), which also keeps NaN pixels
    const bool sky_fin = isfinite(sky);
    const float skyd = __double2float_rd(sky);
    auto counts = [&](float x) { return sky_fin ? !(x <= skyd) : !((double)x - sky <= 0.0); };
    auto value = [&](int k) {  // v of pixel k from the image, 0 where it does not count
        const float x = im[k];
        return counts(x) ? widen(x) - sky : 0.0;
    };
    // first moments
    double m1[3] = {0.0, 0.0, 0.0};
    for (int j = lane; j < W; j += 32) {
        double a0 = 0.0, a1 = 0.0;
#pragma unroll 4
        for (int i = warp; i < H; i += DG_WARPS) {
            const double v = value(i * W + j);
            if (CACHED) cv[i * W + j] = v;
            a0 += v;
            a1 = fma(v, TAB ? dyt[i] : (double)i, a1);
        }
        m1[0] += a0;
        m1[1] = fma((double)j, a0, m1[1]);
        m1[2] += a1;
    }
    block_sums<3>(m1, red);
    // the scalar float64 steps run in one warp (an instruction costs the FP64
    // pipe as much for one lane as for 32) and are shared
    const double s0 = m1[0];
    if (threadIdx.x == 0) {
        sc.x0 = s0 > 0.0 ? m1[1] / s0 : 0.5 * (W - 1);
        sc.y0 = s0 > 0.0 ? m1[2] / s0 : 0.5 * (H - 1);
    }
    __syncthreads();
    const double x0 = sc.x0, y0 = sc.y0;
    for (int i = threadIdx.x; i < (TAB ? H : 0); i += DG_THREADS) {
        const double dy = i - y0;
        dyt[i] = dy;
        dy2t[i] = dy * dy;
        dyf[i] = (float)dy;
    }
    for (int k = threadIdx.x; k < DG_BINS; k += DG_THREADS) hist[k] = 0u;
    __syncthreads();
    // second moments
    double m2[3] = {0.0, 0.0, 0.0};  // xx, yy, xy
    for (int j = lane; j < W; j += 32) {
        double a0 = 0.0, a1 = 0.0, a2 = 0.0;
#pragma unroll 4
        for (int i = warp; i < H; i += DG_WARPS) {
            const double v = CACHED ? cv[i * W + j] : value(i * W + j);
            const double dy = TAB ? dyt[i] : i - y0;
            a0 += v;
            a1 = fma(v, dy, a1);
            a2 = fma(v, TAB ? dy2t[i] : dy * dy, a2);
        }
        const double dx = j - x0;
        m2[0] = fma(dx * dx, a0, m2[0]);
        m2[1] += a2;
        m2[2] = fma(dx, a1, m2[2]);
    }
    block_sums<3>(m2, red);
    if (threadIdx.x == 0) {
        double mxx = m2[0], myy = m2[1], mxy = m2[2];
        if (s0 > 0.0) {
            mxx /= s0;
            myy /= s0;
            mxy /= s0;
        }
        const double tr = mxx + myy, det = mxx * myy - mxy * mxy;
        const double disc = sqrt(fmax(0.25 * tr * tr - det, 0.0));
        const double l1 = 0.5 * tr + disc, l2 = 0.5 * tr - disc;
        const double ax = (l1 > 0.0 && l2 > 0.0) ? sqrt(l2 / l1) : 1.0;
        sc.q = fmin(fmax(ax, 0.05), 1.0);
        double pa = 0.5 * atan2(2.0 * mxy, mxx - myy) * 180.0 / M_PI;
        pa = fmod(pa, 180.0);
        if (pa < 0.0) pa += 180.0;
        s_pa = pa;
        const double th = __ddiv_rn(__dmul_rn(pa, M_PI), 180.0);
        sc.cs = cos(th);
        sc.sn = sin(th);
        sc.csf = (float)sc.cs;
        sc.snf = (float)sc.sn;
        sc.invqf = (float)(1.0 / sc.q);
        s_scale = (float)(268435456.0 / s0);
    }
    __syncthreads();
    // curve of growth: smallest aperture index k in [1, K] with enclosed >= half
    // (K + 1: not reached)
    const double half = 0.5 * s0;
    const int K = 4 * max(H, W);
    int kh;
    if (!(s0 > 0.0) || !isfinite(s0)) {
        kh = s0 == 0.0 ? 1 : K + 1;  // no positive pixel: half = 0; NaN or infinite: never reached
    } else {
        const Ellipse e = sc;
        auto index_at = [&](int i, int j, float dx) {
            return aperture_index(e, i, j, dx, TAB ? dyf[i] : (float)(i - y0), K);
        };
        // enclosed flux below index k and at it, in float64
        auto sums_at = [&](int k, double& below, double& at) {
            double s[2] = {0.0, 0.0};
            for (int j = lane; j < W; j += 32) {
                const float dx = (float)(j - x0);
#pragma unroll 4
                for (int i = warp; i < H; i += DG_WARPS) {
                    if (!CACHED && !counts(im[i * W + j])) continue;
                    const int m = CACHED ? idx[i * W + j] : index_at(i, j, dx);
                    if (m > k) continue;
                    const double v = CACHED ? cv[i * W + j] : value(i * W + j);
                    if (m < k)
                        s[0] += v;
                    else
                        s[1] += v;
                }
            }
            block_sums<2>(s, red);
            below = s[0];
            at = s[1];
        };
        const bool binned = K + 2 <= DG_BINS;
        if (CACHED || binned) {
            // fluxes as integers, 2^28 for the whole: a sum independent of the order
            const float scale = s_scale, skyf = (float)sky;
            for (int j = lane; j < W; j += 32) {
                const float dx = (float)(j - x0);
                for (int i = warp; i < H; i += DG_WARPS) {
                    const float x = im[i * W + j];
                    if (!counts(x)) {
                        if (CACHED) idx[i * W + j] = 0;
                        continue;
                    }
                    const int m = index_at(i, j, dx);
                    if (CACHED) idx[i * W + j] = (unsigned short)m;
                    if (binned) atomicAdd(&hist[m], __float2uint_rz((x - skyf) * scale));
                }
            }
            __syncthreads();
        }
        int lo = 0, hi = K + 1;  // enclosed(lo) < half <= enclosed(hi)
        if (binned) {
            if (warp == 0) {
                // the first bin at which the running sum reaches half the total
                constexpr int PER = (DG_BINS + 31) / 32;
                unsigned mine = 0u;
                for (int t = 0; t < PER; ++t) {
                    const int k = lane * PER + t;
                    if (k < DG_BINS) mine += hist[k];
                }
                unsigned incl = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += u;
                }
                const unsigned want = (__shfl_sync(0xffffffffu, incl, 31) + 1u) / 2u;
                if (lane == 0) s_k = K + 1;
                __syncwarp();
                if (incl >= want && incl - mine < want) {
                    unsigned run = incl - mine;
                    int k = lane * PER;
                    for (; k < min(DG_BINS, lane * PER + PER); ++k) {
                        run += hist[k];
                        if (run >= want) break;
                    }
                    s_k = min(max(k, 1), K + 1);
                }
            }
            __syncthreads();
            const int kg = s_k;
            double below, at;
            sums_at(kg, below, at);
            if (kg <= K) {
                if (below + at >= half)
                    hi = kg;
                else
                    lo = kg;
            }
            if (kg >= 1 && below < half) lo = max(lo, kg - 1);
            if (kg > 1 && !(below < half)) hi = min(hi, kg - 1);
        }
        while (hi - lo > 1) {
            const int km = (lo + hi) >> 1;
            double below, at;
            sums_at(km, below, at);
            if (below + at >= half)
                hi = km;
            else
                lo = km;
        }
        kh = hi;
    }
    if (threadIdx.x == 0) {
        double re = kh <= K ? 0.25 * kh : 1.0;
        re = fmax(re, 0.5);
        const double F = s0 > 0.0 ? s0 : 1.0;
        double* p = out + (long long)b * nslots;
        p[0] = x0;
        p[1] = y0;
        p[2] = F / sersic_flux_e(1.0, re, 2.0, sc.q, kFluxFactorN2);
        p[3] = re;
        p[4] = 2.0;
        p[5] = sc.q;
        p[6] = s_pa;
        p[7] = 0.0;
        p[8] = sky;
    }
}

// ------------------------------------------------------ start selection
// The network's start is taken where every slot is finite and inside its
// bounds and its chi^2 is finite and no larger than the default start's.
__global__ void k_select(int count, int nslots, const double* __restrict__ cand,
                         const double* __restrict__ x2c, const double* __restrict__ dflt,
                         const double* __restrict__ x2d, const double* __restrict__ lo,
                         const double* __restrict__ hi, double* __restrict__ out,
                         int* __restrict__ choice)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= count) return;
    const double* c = cand + (long long)b * nslots;
    bool ok = isfinite(x2c[b]) && (!isfinite(x2d[b]) || x2c[b] <= x2d[b]);
    for (int s = 0; s < nslots; ++s) ok = ok && isfinite(c[s]) && c[s] >= lo[s] && c[s] <= hi[s];
    const double* src = ok ? c : dflt + (long long)b * nslots;
    for (int s = 0; s < nslots; ++s) out[(long long)b * nslots + s] = src[s];
    if (choice) choice[b] = ok ? 1 : 0;
}

}  // namespace

// ================================================================ launchers

size_t cnn_buffers(void* ws, int B, bool training, CnnBuffers* cb)
{
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += (bytes + 255) & ~(size_t)255;
        return at;
    };
    // weight-gradient partials: the first layer's SIMT chunks or layers 2-4's
    // tensor-core chunks, whichever need more
    size_t part = cnn_bwd_tc_part_floats(B);
    {
        const ConvL L = CONV[0];
        const long long total = (long long)B * L.hout * L.hout;
        const long long nchunk = std::min<long long>(std::max<long long>(1, 2048 / (L.cout * L.cin)), total);
        part = std::max(part, (size_t)(nchunk * L.cout * L.cin * 10));
    }
    // the gradient buffers exist only when the call trains
    const size_t T = training ? 1 : 0;
    const size_t wp = take(2ull * NPARAM), wf = take(2ull * CONV_W_END), wb = take(2ull * CONV_W_END),
                 x = take(2ull * B * NPIX), a0 = take(2ull * B * 32 * 32 * 32),
                 a1 = take(2ull * B * 64 * 16 * 16), a2 = take(2ull * B * 64 * 8 * 8),
                 a3 = take(2ull * B * 2048), h = take(4ull * B * 32), y = take(4ull * B * NOUT),
                 gy = take(T * 4ull * B * NOUT), gh = take(T * 4ull * B * 32),
                 g3 = take(T * 4ull * B * 2048), g2 = take(T * 4ull * B * 64 * 8 * 8),
                 g1 = take(T * 4ull * B * 64 * 16 * 16), g0 = take(T * 4ull * B * 32 * 32 * 32),
                 pt = take(T * 4ull * part);
    if (cb && ws) {
        char* p = static_cast<char*>(ws);
        cb->wp = (__nv_bfloat16*)(p + wp);
        cb->wf = (__nv_bfloat16*)(p + wf);
        cb->wb = (__nv_bfloat16*)(p + wb);
        cb->x = (__nv_bfloat16*)(p + x);
        cb->a0 = (__nv_bfloat16*)(p + a0);
        cb->a1 = (__nv_bfloat16*)(p + a1);
        cb->a2 = (__nv_bfloat16*)(p + a2);
        cb->a3 = (__nv_bfloat16*)(p + a3);
        cb->h = (float*)(p + h);
        cb->y = (float*)(p + y);
        cb->gy = (float*)(p + gy);
        cb->gh = (float*)(p + gh);
        cb->g3 = (float*)(p + g3);
        cb->g2 = (float*)(p + g2);
        cb->g1 = (float*)(p + g1);
        cb->g0 = (float*)(p + g0);
        cb->part = (float*)(p + pt);
        cb->part_floats = T * part;
    }
    return o;
}

cudaError_t cnn_prepare(const float* w, const float* x, int B, const CnnBuffers& cb, cudaStream_t s)
{
    k_cast<<<blocks(NPARAM, 256), 256, 0, s>>>(w, cb.wp, cb.wf, cb.wb);
    GF_COUNT_LAUNCH();
    k_to_bf16<<<blocks((long long)B * NPIX, 256), 256, 0, s>>>(x, cb.x, (long long)B * NPIX);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

cudaError_t cnn_forward_fc(const float* w, int B, const CnnBuffers& cb, float* y, cudaStream_t s)
{
    if (B >= 2048)  // (fewer samples leave SMs idle at four a thread)
        k_fc1_fwd<4><<<blocks((long long)(B + 3) / 4 * 32, 256), 256, 0, s>>>(cb.a3, cb.wp, w, cb.h, B);
    else
        k_fc1_fwd<1><<<blocks((long long)B * 32, 128), 128, 0, s>>>(cb.a3, cb.wp, w, cb.h, B);
    GF_COUNT_LAUNCH();
    k_fc2_fwd<<<blocks((long long)B * NOUT, 256), 256, 0, s>>>(cb.h, cb.wp, w, y ? y : cb.y, B);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

cudaError_t cnn_backward(const float* t, int B, float* loss, float* grad, const CnnBuffers& cb,
                         cudaStream_t s)
{
    k_mse<<<1, 256, 0, s>>>(cb.y, t, cb.gy, loss, B);
    GF_COUNT_LAUNCH();
    k_fc2_bwd_w<<<blocks(NOUT * 32 + NOUT, 256), 256, 0, s>>>(cb.gy, cb.h, grad, B);
    GF_COUNT_LAUNCH();
    k_fc2_bwd_x<<<blocks((long long)B * 32, 256), 256, 0, s>>>(cb.gy, cb.h, cb.wp, cb.gh, B);
    GF_COUNT_LAUNCH();
    k_fc1_bwd_w<<<blocks(32 * 2048 + 32, 256), 256, 0, s>>>(cb.gh, cb.a3, grad, B);
    GF_COUNT_LAUNCH();
    k_fc1_bwd_x<<<blocks((long long)B * 2048, 256), 256, 0, s>>>(cb.gh, cb.a3, cb.wp, cb.g3, B);
    GF_COUNT_LAUNCH();
    // layers 4-2 on the tensor cores (weight gradients and the channels-last
    // gradients at the pre-activations of layers 3-1), then layer 1's weights
    float* gout[4] = {cb.g0, cb.g1, cb.g2, cb.g3};
    const __nv_bfloat16* ins[4] = {cb.x, cb.a0, cb.a1, cb.a2};
    cudaError_t e = cnn_backward_tc(B, grad, gout, ins, cb.wf, cb.part, cb.part_floats, s);
    if (e != cudaSuccess) return e;
    const ConvL L = CONV[0];
    const long long total = (long long)B * L.hout * L.hout;
    const int nchunk = (int)std::min<long long>(std::max<long long>(1, 2048 / (L.cout * L.cin)), total);
    static_assert(CONV[0].cin == 1 && CONV[0].cout % WG_CO == 0, "one input channel, whole blocks of outputs");
    k_conv_bwd_w<<<dim3(L.cout / WG_CO, nchunk), WG_THREADS, 0, s>>>(cb.g0, cb.x, cb.part, B, L.hin, L.cout,
                                                                     L.hout, nchunk);
    GF_COUNT_LAUNCH();
    k_conv_bwd_w_sum<<<blocks((long long)L.cout * L.cin * 10, 256), 256, 0, s>>>(cb.part, grad, L.cin, L.cout,
                                                                                nchunk, L.woff, L.boff);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

cudaError_t cnn_adam(float* w, float* m, float* v, const float* g, int step, float lr,
                     cudaStream_t s)
{
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    k_adam<<<blocks(NPARAM, 256), 256, 0, s>>>(w, m, v, g, NPARAM, lr, b1, b2, 1e-8f, c1, c2);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

cudaError_t cnn_init(float* w, unsigned long long seed, cudaStream_t s)
{
    k_init<<<blocks(NPARAM, 256), 256, 0, s>>>(w, seed);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

cudaError_t cnn_input(const float* img, const float* sig, int B, float* x, cudaStream_t s)
{
    k_cnn_input<<<B, 256, 0, s>>>(img, sig, x);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

cudaError_t cnn_encode(const double* params, int nslots, int count, int H, int W, float* t,
                       cudaStream_t s)
{
    k_encode<<<blocks((long long)count * 32, 128), 128, 0, s>>>(params, nslots, count, H, W, t);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

cudaError_t cnn_decode(const float* y, const double* dflt, int count, int H, int W, int flags,
                       double* params, cudaStream_t s)
{
    // one warp per CTA: the b_n solve is a serial FP64 chain per stamp, so it
    // wants the stamps spread over every SM (8,192 stamps: 0.93 ms -> 0.06 ms, with the shorter series)
    k_decode<<<blocks(count, 32), 32, 0, s>>>(y, dflt, count, H, W, flags, params);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

cudaError_t train_sample(unsigned long long seed, int count, double* params, float* psf,
                         int psf_size, cudaStream_t s)
{
    k_train_sample<<<count, 256, 0, s>>>(seed, params, psf, psf_size);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

cudaError_t noise_fill(const float* m, long long n, unsigned long long seed, float sread,
                       float gain, float* d, float* sig, cudaStream_t s)
{
    k_noise<<<blocks(n, 256), 256, 0, s>>>(m, n, seed, sread, gain, d, sig);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

cudaError_t philox_blocks(const unsigned* in, unsigned* out, int n, cudaStream_t s)
{
    k_philox<<<blocks(n, 128), 128, 0, s>>>(in, out, n);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

size_t default_guess_smem(int H, int W)
{
    const int nr = (H == 1 || W == 1) ? H * W : 2 * W + 2 * (H - 2);
    return sizeof(unsigned) * (((size_t)nr + 3) & ~(size_t)3);
}

// pixels per stamp that k_default_guess keeps in shared memory at most (10 bytes
// each, 96 KB: two CTAs per SM; a 64x64 stamp takes 41 KB, four per SM)
constexpr int DG_CACHE_MAX = 9728;

cudaError_t default_guess(int count, const int* H, const int* W, const long long* off,
                          const float* img, double* out, int nslots, size_t smem, int max_npx,
                          int max_rows, cudaStream_t s)
{
    const int ring_cap = (int)(smem / sizeof(unsigned));
    const int cache_cap = max_npx <= DG_CACHE_MAX ? max_npx : 0;
    const size_t bytes = smem + (sizeof(double) + sizeof(unsigned short)) * (size_t)cache_cap;
    auto launch = [&](auto kernel, int* optin) {
        cudaError_t e = ensure_smem_optin((const void*)kernel, (int)bytes, optin);
        if (e != cudaSuccess) return e;
        kernel<<<count, DG_THREADS, bytes, s>>>(H, W, off, img, out, nslots, ring_cap, cache_cap);
        GF_COUNT_LAUNCH();
        return cudaGetLastError();
    };
    static int o0[64], o1[64], o2[64], o3[64];
    if (max_rows <= DG_ROWS)
        return cache_cap ? launch(k_default_guess<true, true>, o0) : launch(k_default_guess<true, false>, o1);
    return cache_cap ? launch(k_default_guess<false, true>, o2) : launch(k_default_guess<false, false>, o3);
}

cudaError_t guess_select(int count, int nslots, const double* cand, const double* x2c,
                         const double* dflt, const double* x2d, const double* lo, const double* hi,
                         double* out, int* choice, cudaStream_t s)
{
    k_select<<<blocks(count, 128), 128, 0, s>>>(count, nslots, cand, x2c, dflt, x2d, lo, hi, out, choice);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

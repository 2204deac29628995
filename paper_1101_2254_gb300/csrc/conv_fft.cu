// conv_fft.cu -- step 2 of the fitting loop in Fourier space (Sec. 3 item 2
// places the PSF convolution there: forward FFTs, a pointwise product, an
// inverse FFT).
//
// The halo-extended grid (He x We) is convolved circularly at a padded size
// Ny x Nx (smallest 2^a 3^b 5^c >= He, and the smallest even one >= We); with
// the PSF wrapped so that its centre sits at (0, 0), the circular result equals
// the direct sum on the valid region, because every output pixel reads only
// grid pixels inside the extended grid.
//
// Extended grids up to 160 x 160 are padded to Nx, Ny in {96, 128, 160} and
// convolved by k_conv_fft_small, one CTA per channel with the half spectrum in
// shared memory (its own comment below).  Larger ones take three passes per
// channel, through shared-memory Stockham or warp register FFTs (fft.cuh,
// warp_fft.cuh), the half spectra held in a global scratch between passes:
//   rows    two real grid rows packed as one complex row, forward FFT, unpacked
//           into the two half spectra (Nx/2 + 1 bins each);
//   columns CPC adjacent spectrum columns per CTA (coalesced), forward FFT along
//           y, product with the PSF spectrum, inverse FFT; only the rows the
//           output needs are written back;
//   rows    inverse of the packing: two half spectra form one complex row, one
//           inverse FFT gives both output rows; only the valid region is kept.
// The PSF spectrum, scaled by 1/(Ny Nx), is computed once per call by the same
// kernels.  Grid rows beyond He are zeros and are never read or written.
#include <math.h>

#include <algorithm>

#include "fft.cuh"
#include "gf_internal.cuh"
#include "conv_fft.cuh"
#include "reg_dft.cuh"
#include "warp_fft.cuh"

namespace {

constexpr int ROW_THREADS = 128;
constexpr int COL_THREADS = 256;
constexpr int COL_UNROLL = 8;   // column-block loads in flight per thread
constexpr int COL_HPRE = 12;    // PSF-spectrum values a thread may hold in registers

__global__ void k_twiddles(int n, float2* tw)
{
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        double s, c;
        sincospi(2.0 * (double)k / (double)n, &s, &c);
        tw[k] = make_float2((float)c, (float)-s);
    }
}

__device__ __forceinline__ void load_tw(float2* dst, const float2* src, int n)
{
    for (int k = threadIdx.x; k < n; k += blockDim.x) dst[k] = src[k];
}

// The wrapped, normalised PSF on the Ny x Nx grid: psf[v][u] / (Ny Nx) at
// ((v - c) mod Ny, (u - c) mod Nx); the grid was zeroed by the caller.
__global__ void k_psf_wrap(FFTArgs f, int count, const StampInfo* st, const float* psf)
{
    const int b = blockIdx.x >> 3, part = blockIdx.x & 7;  // 8 CTAs per stamp
    if (b >= count) return;
    const int P = st[b].P, c = st[b].c;
    const float scale = (float)(1.0 / ((double)f.Ny * (double)f.Nx));
    float* g = f.psfgrid + (long long)b * f.Ny * f.Nx;
    const float* p = psf + st[b].psf_off;
    for (int t = part * blockDim.x + threadIdx.x; t < P * P; t += 8 * blockDim.x) {
        const int v = t / P, u = t - v * P;
        const int y = ((v - c) % f.Ny + f.Ny) % f.Ny, x = ((u - c) % f.Nx + f.Nx) % f.Nx;
        g[(long long)y * f.Nx + x] = p[t] * scale;
    }
}

// Forward row pass.  Problem p = blockIdx.x / io.nblk covers one real grid (rows `rows`
// valid of row stride `ld`, `width` valid columns) and one half-spectrum array
// (Kx = Nx/2 + 1 bins per row).  Block x of the problem handles rows 2x and 2x + 1.
// (Every FFT pass numbers its CTAs problem-major in one grid dimension: a
// problem count of count * channels may exceed the 65,535 of the y dimension.)
__global__ void __launch_bounds__(ROW_THREADS) k_fft_rows_fwd(FFTArgs f, RowIO io, PassArgs a)
{
    pdl_entry();
    extern __shared__ __align__(16) float2 sm[];
    const int p = blockIdx.x / io.nblk, bx = blockIdx.x - p * io.nblk;
    if (a.lm && a.lm[p / io.nchan].phase != a.phase) return;
    const int Nx = f.Nx, Kx = Nx / 2 + 1;
    float2* bufA = sm;
    float2* bufB = sm + Nx;
    float2* tw = sm + 2 * Nx;
    load_tw(tw, f.tw_x, Nx);
    const int y0 = 2 * bx, y1 = y0 + 1;
    const float* in = io.in + (long long)p * io.in_stride;
    for (int x = threadIdx.x; x < Nx; x += blockDim.x) {
        const bool cx = x < io.width;
        const float va = (cx && y0 < io.rows) ? in[(long long)y0 * io.ld + x] : 0.0f;
        const float vb = (cx && y1 < io.rows) ? in[(long long)y1 * io.ld + x] : 0.0f;
        bufA[x] = make_float2(va, vb);
    }
    __syncthreads();
    const float2* Z = fft_smem(f.px, bufA, bufB, 0, tw, -1.0f);
    float2* out = io.spec + (long long)p * io.spec_stride;
    for (int k = threadIdx.x; k < Kx; k += blockDim.x) {
        const float2 zk = Z[k], zm = cconj(Z[(Nx - k) % Nx]);
        const float2 s = cadd(zk, zm), d = csub(zk, zm);
        // A = (Z[k] + conj Z[N-k]) / 2,  B = (Z[k] - conj Z[N-k]) / (2i)
        if (y0 < io.out_rows) out[(long long)y0 * Kx + k] = make_float2(0.5f * s.x, 0.5f * s.y);
        if (y1 < io.out_rows) out[(long long)y1 * Kx + k] = make_float2(0.5f * d.y, -0.5f * d.x);
    }
    if (a.work && threadIdx.x == 0) atomicAdd(&a.work[PROF_CONV], (unsigned long long)f.flops_row);
}

// Column pass.  mode 0: forward only, all Ny rows written (the PSF spectrum);
// mode 1: forward, product with the PSF spectrum, inverse, rows [c, c + H)
// written back in place.
__global__ void __launch_bounds__(COL_THREADS) k_fft_cols(FFTArgs f, ColIO io, PassArgs a, int mode)
{
    pdl_entry();
    extern __shared__ __align__(16) float2 sm[];
    const int p = blockIdx.x / io.nblk, bx = blockIdx.x - p * io.nblk;
    const int b = p / io.nchan;
    if (a.lm && a.lm[b].phase != a.phase) return;
    const int Ny = f.Ny, Kx = f.Nx / 2 + 1, B = f.cpc, logB = __ffs(B) - 1;  // B a power of two
    float2* bufA = sm;
    float2* bufB = sm + Ny * B;
    float2* tw = sm + 2 * Ny * B;
    load_tw(tw, f.tw_y, Ny);
    const int kx0 = bx * B;
    float2* spec = io.spec + (long long)p * io.spec_stride;
    const int total = Ny * B;
    // the column block: eight loads per thread in flight before their stores
    for (int t0 = threadIdx.x; t0 < total; t0 += COL_UNROLL * COL_THREADS) {
        float2 v[COL_UNROLL];
#pragma unroll
        for (int u = 0; u < COL_UNROLL; ++u) {
            const int t = t0 + u * COL_THREADS;
            const int y = t >> logB, kx = kx0 + (t & (B - 1));
            v[u] = (t < total && y < io.rows_in && kx < Kx) ? spec[(long long)y * Kx + kx]
                                                            : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < COL_UNROLL; ++u) {
            const int t = t0 + u * COL_THREADS;
            if (t < total) bufA[t] = v[u];
        }
    }
    // the PSF spectrum this thread multiplies, fetched now so that its latency
    // hides behind the forward transform (when it fits the registers)
    const float2* Hs = f.hhat + (long long)b * Ny * Kx;
    float2 hv[COL_HPRE];
    const bool hpre = mode == 1 && total <= COL_HPRE * COL_THREADS;
    if (hpre) {
#pragma unroll
        for (int u = 0; u < COL_HPRE; ++u) {
            const int t = threadIdx.x + u * COL_THREADS;
            const int y = t >> logB, kx = kx0 + (t & (B - 1));
            hv[u] = (t < total && kx < Kx) ? Hs[(long long)y * Kx + kx] : make_float2(0.f, 0.f);
        }
    }
    __syncthreads();
    float2* X = fft_smem(f.py, bufA, bufB, logB, tw, -1.0f);
    if (a.work && threadIdx.x == 0) atomicAdd(&a.work[PROF_CONV], (unsigned long long)f.flops_col);
    if (mode == 0) {
        for (int t = threadIdx.x; t < Ny * B; t += blockDim.x) {
            const int y = t >> logB, kx = kx0 + (t & (B - 1));
            if (kx < Kx) spec[(long long)y * Kx + kx] = X[t];
        }
        return;
    }
    if (hpre) {
#pragma unroll
        for (int u = 0; u < COL_HPRE; ++u) {
            const int t = threadIdx.x + u * COL_THREADS;
            const int kx = kx0 + (t & (B - 1));
            if (t < total && kx < Kx) X[t] = cmul(X[t], hv[u]);
        }
    } else {
        for (int t = threadIdx.x; t < total; t += blockDim.x) {
            const int y = t >> logB, kx = kx0 + (t & (B - 1));
            if (kx < Kx) X[t] = cmul(X[t], Hs[(long long)y * Kx + kx]);
        }
    }
    __syncthreads();
    float2* other = (X == bufA) ? bufB : bufA;
    const float2* Yv = fft_smem(f.py, X, other, logB, tw, 1.0f);
    const int r0 = io.row0, r1 = io.row0 + io.nrows_out;
    for (int t = threadIdx.x; t < Ny * B; t += blockDim.x) {
        const int y = t >> logB, kx = kx0 + (t & (B - 1));
        if (kx < Kx && y >= r0 && y < r1) spec[(long long)y * Kx + kx] = Yv[t];
    }
}

// Inverse row pass: output rows 2x, 2x + 1 of an H x W result from spectrum
// rows row0 + 2x, row0 + 2x + 1; grid columns [col0, col0 + W) are kept.
__global__ void __launch_bounds__(ROW_THREADS) k_fft_rows_inv(FFTArgs f, RowInvIO io, PassArgs a)
{
    pdl_entry();
    extern __shared__ __align__(16) float2 sm[];
    const int p = blockIdx.x / io.nblk, bx = blockIdx.x - p * io.nblk;
    if (a.lm && a.lm[p / io.nchan].phase != a.phase) return;
    const int Nx = f.Nx, Kx = Nx / 2 + 1;
    float2* bufA = sm;
    float2* bufB = sm + Nx;
    float2* tw = sm + 2 * Nx;
    load_tw(tw, f.tw_x, Nx);
    const int i0 = 2 * bx, i1 = i0 + 1;
    const bool has1 = i1 < io.H;
    const float2* spec = io.spec + (long long)p * io.spec_stride;
    const float2* sa = spec + (long long)(io.row0 + i0) * Kx;
    const float2* sb = spec + (long long)(io.row0 + i1) * Kx;
    for (int k = threadIdx.x; k < Nx; k += blockDim.x) {
        float2 A, Bv;
        if (k < Kx) {
            A = sa[k];
            Bv = has1 ? sb[k] : make_float2(0.f, 0.f);
        } else {
            A = cconj(sa[Nx - k]);
            Bv = has1 ? cconj(sb[Nx - k]) : make_float2(0.f, 0.f);
        }
        bufA[k] = make_float2(A.x - Bv.y, A.y + Bv.x);  // A + i B
    }
    __syncthreads();
    const float2* z = fft_smem(f.px, bufA, bufB, 0, tw, 1.0f);
    float* out = io.out + (long long)p * io.out_stride;
    for (int j = threadIdx.x; j < io.W; j += blockDim.x) {
        const float2 v = z[io.col0 + j];
        out[(long long)i0 * io.W + j] = v.x;
        if (has1) out[(long long)i1 * io.W + j] = v.y;
    }
    if (a.work && threadIdx.x == 0) atomicAdd(&a.work[PROF_CONV], (unsigned long long)f.flops_row);
}

// ---------------------------------------------------------- warp row passes
// For Nx = 32 M with M in the WarpFFTFactor list the row passes use one warp
// per pair of rows and the register FFT of warp_fft.cuh: no block barrier
// between stages, every input load of a lane issued before the first
// butterfly.  The CTA's four warps share the padded twiddle table; each warp
// has an Nx-element buffer to bring its result into natural order (and, in the
// forward pass, to pair Z[k] with Z[Nx - k] for the unpacking).
constexpr int WROW_WARPS = 4;

template <int M>
__global__ void __launch_bounds__(WROW_WARPS * 32) k_fft_rows_fwd_w(FFTArgs f, RowIO io, PassArgs a)
{
    pdl_entry();
    constexpr int N = 32 * M, Kx = N / 2 + 1;
    extern __shared__ __align__(16) float2 sm[];
    const int p = blockIdx.x / io.nblk, bx = blockIdx.x - p * io.nblk;
    if (a.lm && a.lm[p / io.nchan].phase != a.phase) return;
    float2* tws = sm;
    for (int t = threadIdx.x; t < N; t += blockDim.x) tws[warp_fft_pad(t)] = f.tw_x[t];
    __syncthreads();
    const int warp = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int y0 = 2 * (bx * WROW_WARPS + warp), y1 = y0 + 1;
    if (y0 >= io.out_rows) return;
    const float* in = io.in + (long long)p * io.in_stride;
    float2 v[M];
#pragma unroll
    for (int j = 0; j < M; ++j) {
        const int x = l + 32 * j;
        const bool cx = x < io.width;
        const float va = (cx && y0 < io.rows) ? in[(long long)y0 * io.ld + x] : 0.0f;
        const float vb = (cx && y1 < io.rows) ? in[(long long)y1 * io.ld + x] : 0.0f;
        v[j] = make_float2(va, vb);
    }
    warp_fft<M, false>(v, tws);
    float2* z = sm + warp_fft_table_len(N) + warp * N;
    const int br = bitrev5(l);
#pragma unroll
    for (int k2 = 0; k2 < M; ++k2) z[k2 + M * br] = v[k2];
    __syncwarp();
    float2* out = io.spec + (long long)p * io.spec_stride;
    for (int k = l; k < Kx; k += 32) {
        const float2 zk = z[k], zm = cconj(z[(N - k) % N]);
        const float2 s = cadd(zk, zm), d = csub(zk, zm);
        // A = (Z[k] + conj Z[N-k]) / 2,  B = (Z[k] - conj Z[N-k]) / (2i)
        out[(long long)y0 * Kx + k] = make_float2(0.5f * s.x, 0.5f * s.y);
        if (y1 < io.out_rows) out[(long long)y1 * Kx + k] = make_float2(0.5f * d.y, -0.5f * d.x);
    }
    if (a.work && l == 0) atomicAdd(&a.work[PROF_CONV], (unsigned long long)f.flops_row);
}

template <int M>
__global__ void __launch_bounds__(WROW_WARPS * 32) k_fft_rows_inv_w(FFTArgs f, RowInvIO io, PassArgs a)
{
    pdl_entry();
    constexpr int N = 32 * M, Kx = N / 2 + 1;
    extern __shared__ __align__(16) float2 sm[];
    const int p = blockIdx.x / io.nblk, bx = blockIdx.x - p * io.nblk;
    if (a.lm && a.lm[p / io.nchan].phase != a.phase) return;
    float2* tws = sm;
    for (int t = threadIdx.x; t < N; t += blockDim.x) tws[warp_fft_pad(t)] = f.tw_x[t];
    __syncthreads();
    const int warp = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int i0 = 2 * (bx * WROW_WARPS + warp), i1 = i0 + 1;
    if (i0 >= io.H) return;
    const bool has1 = i1 < io.H;
    const float2* spec = io.spec + (long long)p * io.spec_stride;
    const float2* sa = spec + (long long)(io.row0 + i0) * Kx;
    const float2* sb = spec + (long long)(io.row0 + i1) * Kx;
    float2 v[M];
#pragma unroll
    for (int j = 0; j < M; ++j) {
        const int k = l + 32 * j;
        float2 A, Bv;
        if (k < Kx) {
            A = sa[k];
            Bv = has1 ? sb[k] : make_float2(0.f, 0.f);
        } else {
            A = cconj(sa[N - k]);
            Bv = has1 ? cconj(sb[N - k]) : make_float2(0.f, 0.f);
        }
        v[j] = make_float2(A.x - Bv.y, A.y + Bv.x);  // A + i B
    }
    warp_fft<M, true>(v, tws);
    float2* z = sm + warp_fft_table_len(N) + warp * N;
    const int br = bitrev5(l);
#pragma unroll
    for (int k2 = 0; k2 < M; ++k2) z[k2 + M * br] = v[k2];
    __syncwarp();
    float* out = io.out + (long long)p * io.out_stride;
    for (int j = l; j < io.W; j += 32) {
        const float2 w = z[io.col0 + j];
        out[(long long)i0 * io.W + j] = w.x;
        if (has1) out[(long long)i1 * io.W + j] = w.y;
    }
    if (a.work && l == 0) atomicAdd(&a.work[PROF_CONV], (unsigned long long)f.flops_row);
}

// ------------------------------------------- one CTA per transform (small grids)
// For Nx = 8 MX and Ny = 8 MY with MX, MY in {12, 16, 20} (grids up to 160 x 160)
// the whole convolution of one channel tile runs in one CTA: its half spectrum
// (Ny x Kx complex values, at most 104 KB) stays in shared memory between the
// three stages, so the only global traffic is the grid read, the PSF spectrum
// read and the valid region written (in an LM trial pass, the image and sigma
// read and the chi^2 partials of the 16 x 32 output blocks written instead of
// the region).
// The tile is the whole stamp where its grid fits (the FFT method), or
// toy x tox outputs of a stamp of any size (the tiled method, overlap-save: the
// tile's grid window is toy + P - 1 by tox + P - 1, at most Ny x Nx; toy and tox
// are multiples of the 16 x 32 blocks of the trial partials).
// The grid is persistent over the (tile, channel) items of the pass's work list,
// channels innermost: the twiddle tables are built once per CTA, a stamp's PSF
// spectrum is met by its channels one after the other, and stamps that have
// left the LM loop cost nothing.
//
// What bounds it is instruction issue, so the transforms are split to need few:
// a length-8M transform is an M-point DFT per residue n mod 8 (phase A) and an
// 8-point DFT per k mod M (phase B), each in one thread's registers
// (reg_dft.cuh), exchanged once through shared memory in place, with one
// twiddle product between them:
//   X[k2 + M k1] = sum_{n1 < 8} w_8^{n1 k1} w_N^{n1 k2} sum_{n2 < M} x[n1 + 8 n2] w_M^{n2 k2}
// (the inverse runs B, then A).  About 19 operations a value and transform,
// packed two to an instruction where they are additions.  The stages:
//   rows     A on pairs of grid rows packed as one complex row, straight from
//            global memory; B on the classes k2 and M - k2 together, whose
//            outputs are each other's mirror images, so the two half spectra are
//            unpacked in registers;
//   columns  A; B, product with the PSF spectrum and the inverse B in one go; A;
//   rows     the packing and B; A, whose outputs go to global memory (a trial
//            pass brings them through shared memory, a warp per row pair).
// A thread's row index and column advance so that the column phases touch
// consecutive addresses; the row phases exchange through the pair's own two
// spectrum rows at an odd stride (pair p of a group at p (Nx + 1), residue n1 at
// 2 n1), free of bank conflicts.
// The PSF spectrum is made by the same kernel (psf_mode): the PSF, read wrapped
// and scaled, through the row phases and the forward column phases, stored as
// hperm[k1][k2][kx] for ky = k2 + MY k1, the order in which phase B reads it.
// Against the warp-shuffle transform (a warp per row pair or column, radix-2
// stages by shuffles) that stood here: 21.7 against 40.8 thousand warp
// instructions a transform, issued at 42 against 84 % (24 warps an SM and a
// barrier a phase), so that alone it is not faster (Jacobian pass of 8,192 stamps
// of 64x64, 57,344 transforms of 96x96: 2.16 ms then, 2.3 now); but as a
// persistent kernel over the work list the passes of 8,192 fits' loop take 15.3 ms
// for 17.0, and 512 fits of 48-256 px stamps 11.6 ms for 14.5.
// threads: a group's phase B needs 16 MX of them.  Four CTAs of 192 (80 registers
// each, 24 warps an SM) measured faster than four of 256 (64, spilling) and five
// of 192 (64): 42.4, 43.8 and 47.1 ms on 8,192 fits of 64x64 stamps.
constexpr int small_threads(int MX) { return 16 * MX; }

struct SmallIO {
    int toy, tox;         // outputs of a tile (a multiple of 16 x 32, or the stamp's H x W)
    int one_tile;         // every stamp is one tile
    const StampInfo* st;
    const float* psf;     // psf_mode: the PSFs and their scale 1 / (4 Ny Nx)
    float scale;
    float2* hperm;        // per stamp Kx * Ny values (written in psf_mode)
    int count;            // stamps (psf_mode)
    int psf_mode;
    float flops;          // a full tile's transform work (profiling)
};

// One (tile, channel) item as its CTA sees it, in shared memory: the phases read
// what they need of it instead of carrying it in registers, and one thread
// fills the next item's while the current one is transformed.
struct TileItem {
    const float* in;        // the grid window (or, in psf_mode, the PSF)
    const float* img;       // the tile's image and sigma
    const float* sig;
    float* out;             // the tile's outputs
    float2* hp;             // the stamp's PSF spectrum
    long long slot;         // the tile's first trial partial
    int W, We, c, P;        // the stamp's width, its grid's, (P - 1) / 2, P
    int hO, wO;             // the tile's outputs
    int rows, width;        // its grid window
    int npair, ngrp, G;     // row pairs of the window, their exchange groups and a group's pairs
    int ngo, Go;            // the same for the output rows
    int ch;
    int psf_mode;
    float scale;            // psf_mode: the PSF's
    float tmw, tmsky;       // a trial channel's weight and sky
};

// most row pairs of one exchange group: a thread per pair and class in phase B
constexpr int SMALL_GROUP = 32;

constexpr size_t small_smem(int MX, int MY)
{
    // the half spectrum, the twiddle tables (rows of M + 1), the trial pass's
    // row-pair sums per 32 columns
    return sizeof(float2) * ((size_t)(8 * MY) * (4 * MX + 1) + 8 * (size_t)(MX + 1) + 8 * (size_t)(MY + 1) +
                             (size_t)(4 * MY) * ((8 * MX) / 32)) + 2 * sizeof(TileItem);
}

// CTAs per SM that the kernel's shared memory allows (227 KB per SM, 1 KB of
// it taken by each CTA), at most four, which its register budget is held to
template <int MX, int MY>
constexpr int small_ctas_per_sm()
{
    const int n = (int)((227u * 1024u) / (small_smem(MX, MY) + 1024));
    return n < 1 ? 1 : (n > 4 ? 4 : n);
}

// The phases of k_conv_fft_small, separated by barriers.
template <int MX, int MY>
struct TilePhases {
    static constexpr int Nx = 8 * MX, Ny = 8 * MY, Kx = Nx / 2 + 1, NT = small_threads(MX);
    static constexpr int HJ = MX / 2;  // class pairs of a row transform
    static_assert(MX % 2 == 0 && MY % 2 == 0 && 2 * Kx > Nx && NT / HJ >= SMALL_GROUP,
                  "the exchange fits the pair's rows, a group the block");

    // slot of Y[n1][k2] in a pair's exchange area
    static __device__ __forceinline__ int pos(int n1, int k2) { return (k2 >> 1) * 16 + 2 * n1 + (k2 & 1); }

    // rows, phase A: pairs (y0, y0 + 1) of the grid window; rows >= rows are zeros
    static __device__ __forceinline__ void rows_a(float2* spec, const float2* twx, const TileItem& I)
    {
#pragma unroll 1
        for (int t = (int)threadIdx.x; t < 8 * I.npair; t += NT) {
            const int pr = t >> 3, n1 = t & 7;
            const int y0 = 2 * pr, y1 = y0 + 1;
            float2 v[MX];
            if (I.psf_mode) {  // psf[v][u] scale at ((v - c) mod Ny, (u - c) mod Nx)
                const int P = I.P, c = I.c;
                const float* in = I.in;
                const int v0 = y0 <= c ? y0 + c : y0 + c - Ny, v1 = y1 <= c ? y1 + c : y1 + c - Ny;
#pragma unroll
                for (int n2 = 0; n2 < MX; ++n2) {
                    const int x = n1 + 8 * n2, u = x <= c ? x + c : x + c - Nx;
                    v[n2].x = u >= 0 && v0 >= 0 ? in[v0 * P + u] * I.scale : 0.0f;
                    v[n2].y = u >= 0 && v1 >= 0 ? in[v1 * P + u] * I.scale : 0.0f;
                }
            } else {
                const int We = I.We, width = I.width;
                const float* r0 = I.in + (long long)y0 * We + n1;
                const bool two = y1 < I.rows;
#pragma unroll
                for (int n2 = 0; n2 < MX; ++n2) {
                    const bool cx = n1 + 8 * n2 < width;
                    v[n2].x = cx ? r0[8 * n2] : 0.0f;
                    v[n2].y = cx && two ? r0[We + 8 * n2] : 0.0f;
                }
            }
            rdft<MX, false>(v);
            const int G = I.G;
            float2* e = spec + (pr / G) * (2 * G * Kx) + (pr % G) * (Nx + 1);
            const float2* w = twx + n1 * (MX + 1);
            e[pos(n1, 0)] = v[0];
#pragma unroll
            for (int k2 = 1; k2 < MX; ++k2) e[pos(n1, k2)] = c_mul(v[k2], w[k2]);
        }
    }

    // rows, phase B and unpacking: with Z = A + i B (rows y0 and y1) the bins are
    // A = Z[k] + conj Z[N-k], B = (Z[k] - conj Z[N-k]) / i, twice the spectra
    // (the PSF's scale has the factor)
    static __device__ __forceinline__ void rows_b(float2* spec, const TileItem& I)
    {
#pragma unroll 1
        for (int g = 0; g < I.ngrp; ++g) {
            const int G = I.G, np = min(G, I.npair - g * G);
            const int t0 = (int)threadIdx.x, j = t0 / np, p = t0 - j * np;
            const int jb = j == 0 ? HJ : MX - j;
            float2 za[8], zb[8];
            if (j < HJ) {
                const float2* e = spec + g * (2 * G * Kx) + p * (Nx + 1);
#pragma unroll
                for (int n1 = 0; n1 < 8; ++n1) {
                    za[n1] = e[pos(n1, j)];
                    zb[n1] = e[pos(n1, jb)];
                }
            }
            __syncthreads();
            if (j < HJ) {
                rdft8<false>(za);
                rdft8<false>(zb);
                float2* sa = spec + (g * G + p) * (2 * Kx);
                auto unpack = [&](int k, float2 zk, float2 zm) {
                    sa[k] = c2(zk.x + zm.x, zk.y - zm.y);
                    sa[Kx + k] = c2(zk.y + zm.y, zm.x - zk.x);
                };
                // the mirror of (k1, j) is (7 - k1, MX - j), but the classes 0 and MX / 2
                // mirror themselves
#pragma unroll
                for (int k1 = 0; k1 < 4; ++k1) {
                    unpack(j + MX * k1, za[k1], j == 0 ? za[(8 - k1) % 8] : zb[7 - k1]);
                    unpack(jb + MX * k1, zb[k1], j == 0 ? zb[7 - k1] : za[7 - k1]);
                }
                if (j == 0) unpack(4 * MX, za[4], za[4]);
            }
        }
    }

    // columns, phase A: value (n1 + 8 n2, k) sits at t + 8 Kx n2 for t = n1 Kx + k
    static __device__ __forceinline__ void cols_a(float2* spec, const float2* twy, const TileItem& I)
    {
#pragma unroll 1
        for (int t = (int)threadIdx.x; t < 8 * Kx; t += NT) {
            const int n1 = t / Kx, hw = 2 * I.npair;
            float2* col = spec + t;
            float2 v[MY];
#pragma unroll
            for (int n2 = 0; n2 < MY; ++n2)
                v[n2] = n1 + 8 * n2 < hw ? col[8 * Kx * n2] : c2(0.0f, 0.0f);
            rdft<MY, false>(v);
            const float2* w = twy + n1 * (MY + 1);
            col[0] = v[0];
#pragma unroll
            for (int k2 = 1; k2 < MY; ++k2) col[8 * Kx * k2] = c_mul(v[k2], w[k2]);
        }
    }

    // columns, phase B, the PSF product and the inverse's phase B
    static __device__ __forceinline__ void cols_b(float2* spec, const TileItem& I)
    {
#pragma unroll 1
        for (int t = (int)threadIdx.x; t < MY * Kx; t += NT) {
            float2* col = spec + (t / Kx) * (8 * Kx) + t % Kx;
            float2* hp = I.hp + t;
            float2 v[8], h[8];
            if (!I.psf_mode) {
#pragma unroll
                for (int k1 = 0; k1 < 8; ++k1) h[k1] = hp[k1 * (MY * Kx)];
            }
#pragma unroll
            for (int n1 = 0; n1 < 8; ++n1) v[n1] = col[n1 * Kx];
            rdft8<false>(v);
            if (I.psf_mode) {
#pragma unroll
                for (int k1 = 0; k1 < 8; ++k1) hp[k1 * (MY * Kx)] = v[k1];
                continue;
            }
#pragma unroll
            for (int k1 = 0; k1 < 8; ++k1) v[k1] = c_mul(v[k1], h[k1]);
            rdft8<true>(v);
#pragma unroll
            for (int n1 = 0; n1 < 8; ++n1) col[n1 * Kx] = v[n1];
        }
    }

    // columns, the inverse's phase A; the rows [c, c + hO) are kept
    static __device__ __forceinline__ void cols_ai(float2* spec, const float2* twy, const TileItem& I)
    {
#pragma unroll 1
        for (int t = (int)threadIdx.x; t < 8 * Kx; t += NT) {
            const int n1 = t / Kx, lo = I.c, hi = I.c + I.hO;
            float2* col = spec + t;
            const float2* w = twy + n1 * (MY + 1);
            float2 v[MY];
            v[0] = col[0];
#pragma unroll
            for (int k2 = 1; k2 < MY; ++k2) v[k2] = c_mulc(col[8 * Kx * k2], w[k2]);
            rdft<MY, true>(v);
#pragma unroll
            for (int n2 = 0; n2 < MY; ++n2) {
                const int y = n1 + 8 * n2;
                if (y >= lo && y < hi) col[8 * Kx * n2] = v[n2];
            }
        }
    }

    // output rows of group g (np pairs): the packing Z = A + i B of rows (i0, i0 + 1)
    // and the inverse's phase B
    static __device__ __forceinline__ void out_b(float2* area, const TileItem& I, int g, int np)
    {
        const int t0 = (int)threadIdx.x, j = t0 / np, p = t0 - j * np;
        const int jb = j == 0 ? HJ : MX - j;
        float2 za[8], zb[8];
        if (j < HJ) {
            const float2* sa = area + p * (2 * Kx);
            const bool has1 = 2 * (g * I.Go + p) + 1 < I.hO;
            auto pack = [&](int k, float2& zk, float2& zm) {  // Z[k] and Z[N - k]
                const float2 A = sa[k], B = has1 ? sa[Kx + k] : c2(0.0f, 0.0f);
                zk = c2(A.x - B.y, A.y + B.x);
                zm = c2(A.x + B.y, B.x - A.y);
            };
            // (k1, j) and its mirror, as in the unpacking
            float2 ma[4], mb[4], mid = c2(0.0f, 0.0f), drop;
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) {
                pack(j + MX * k1, za[k1], ma[k1]);
                pack(jb + MX * k1, zb[k1], mb[k1]);
            }
            if (j == 0) pack(4 * MX, mid, drop);
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) {
                za[7 - k1] = j != 0 ? mb[k1] : k1 < 3 ? ma[(k1 + 1) % 4] : mid;
                zb[7 - k1] = j != 0 ? ma[k1] : mb[k1];
            }
            rdft8<true>(za);
            rdft8<true>(zb);
        }
        __syncthreads();
        if (j < HJ) {
            float2* e = area + p * (Nx + 1);
#pragma unroll
            for (int n1 = 0; n1 < 8; ++n1) {
                e[pos(n1, j)] = za[n1];
                e[pos(n1, jb)] = zb[n1];
            }
        }
        __syncthreads();
    }

    // and the inverse's phase A: the outputs to global memory, or (a trial pass) each
    // pair's two rows of floats in place of its exchange area
    static __device__ __forceinline__ void out_a(float2* area, const float2* twx, const TileItem& I, int g, int np, int trial)
    {
        // phase A: a thread per pair and residue
#pragma unroll 1
        for (int t = (int)threadIdx.x; t - (t & 31) < 8 * np; t += NT) {  // whole warps: a pair's eight threads share one
            const int pa = t >> 3, n1 = t & 7;
            float2* e = area + pa * (Nx + 1);
            float2 v[MX];
            if (pa < np) {
                const float2* w = twx + n1 * (MX + 1);
                v[0] = e[pos(n1, 0)];
#pragma unroll
                for (int k2 = 1; k2 < MX; ++k2) v[k2] = c_mulc(e[pos(n1, k2)], w[k2]);
                rdft<MX, true>(v);
            }
            if (!trial) {
                if (pa < np) {
                    const int i0 = 2 * (g * I.Go + pa), c = I.c, W = I.W, wO = I.wO;
                    float* o0 = I.out + (long long)i0 * W + n1 - c;
                    const bool has1 = i0 + 1 < I.hO;
#pragma unroll
                    for (int n2 = 0; n2 < MX; ++n2) {
                        const int jx = n1 + 8 * n2 - c;
                        if (jx >= 0 && jx < wO) {
                            o0[8 * n2] = v[n2].x;
                            if (has1) o0[W + 8 * n2] = v[n2].y;
                        }
                    }
                }
                continue;
            }
            __syncwarp();  // the pair's exchange area becomes its two rows of floats
            if (pa < np) {
                float* rowsf = reinterpret_cast<float*>(e);
#pragma unroll
                for (int n2 = 0; n2 < MX; ++n2) {
                    rowsf[n1 + 8 * n2] = v[n2].x;
                    rowsf[Nx + n1 + 8 * n2] = v[n2].y;
                }
            }
        }
    }

    // a trial pass: each row pair's chi^2 per 32 columns
    static __device__ __forceinline__ void out_chi2(const float2* area, CSum* part, const TileItem& I, int g, int np)
    {
        const int warp = threadIdx.x >> 5, l = threadIdx.x & 31;
        const int hO = I.hO, wO = I.wO, W = I.W, c = I.c, nbx = (wO + 31) / 32;
        const float tmw = I.tmw, tmsky = I.tmsky;
        const float* img = I.img;
        const float* sig = I.sig;
#pragma unroll 1
        for (int q = warp; q < np; q += NT / 32) {
            const float* rowsf = reinterpret_cast<const float*>(area + q * (Nx + 1)) + c;
            const int r0 = 2 * (g * I.Go + q);
#pragma unroll 1
            for (int t = 0; t < nbx; ++t) {
                const int jx = l + 32 * t;
                CSum cs = {0.0f, 0.0f};
                if (jx < wO) {
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        if (r == 1 && r0 + 1 >= hO) break;
                        const long long px = (long long)(r0 + r) * W + jx;
                        const float d = __ldg(&img[px]), sg = __ldg(&sig[px]);
                        if (isfinite(d) && isfinite(sg) && sg > 0.0f) {
                            const float m = rowsf[r * Nx + jx];
                            const float zr = (d - fmaf(tmw, m, tmsky)) / sg;
                            csum_add(cs, zr * zr);
                        }
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    CSum other;
                    other.s = __shfl_down_sync(0xffffffffu, cs.s, o);
                    other.c = __shfl_down_sync(0xffffffffu, cs.c, o);
                    cs = csum_merge(cs, other);
                }
                if (l == 0) part[(g * I.Go + q) * nbx + t] = cs;
            }
        }
    }
};

template <int MX, int MY>
__global__ void __launch_bounds__(small_threads(MX), small_ctas_per_sm<MX, MY>()) k_conv_fft_small(
    const __grid_constant__ SmallIO io, const __grid_constant__ PassArgs a, const float2* tw_x, const float2* tw_y)
{
    pdl_entry();
    constexpr int Nx = 8 * MX, Ny = 8 * MY, Kx = Nx / 2 + 1, NT = small_threads(MX);
    constexpr int HJ = MX / 2;    // class pairs of a row transform
    using Ph = TilePhases<MX, MY>;
    static_assert(sizeof(CSum) == sizeof(float2), "a partial takes one float2 slot");
    extern __shared__ __align__(16) float2 sm[];
    float2* spec = sm;                    // Ny rows of stride Kx (odd)
    float2* twx = spec + Ny * Kx;         // w_Nx^{n1 k2} at n1 (MX + 1) + k2
    float2* twy = twx + 8 * (MX + 1);     // w_Ny^{n1 k2} at n1 (MY + 1) + k2
    CSum* part = reinterpret_cast<CSum*>(twy + 8 * (MY + 1));
    TileItem* info = reinterpret_cast<TileItem*>(part + 4 * MY * (Nx / 32));
    const int tid = threadIdx.x;
    for (int t = tid; t < 8 * MX; t += NT) twx[(t / MX) * (MX + 1) + t % MX] = tw_x[(t / MX) * (t % MX)];
    for (int t = tid; t < 8 * MY; t += NT) twy[(t / MY) * (MY + 1) + t % MY] = tw_y[(t / MY) * (t % MY)];
    const int nchan = io.psf_mode ? 1 : a.nchan;
    const int n = io.psf_mode ? io.count : *a.wl.n;
    const int* pre = io.psf_mode ? nullptr : a.wl.pre + WK_CONV * (a.count + 1);
    const long long items = (long long)(io.one_tile ? n : pre[n]) * nchan;
    // this CTA's share, spread evenly
    const long long it0 = items * blockIdx.x / gridDim.x, it1 = items * (blockIdx.x + 1) / gridDim.x;
    int hint = -1;
    auto fill = [&](long long it, TileItem& q) {
        const int tile = (int)(it / nchan), ch = (int)(it - (long long)tile * nchan);
        const int li = io.one_tile ? tile : wl_locate(pre, n, tile, hint);
        const int b = io.psf_mode ? tile : a.wl.ids[li];
        const StampInfo& st = io.st[b];
        int ty0 = 0, tx0 = 0;
        if (!io.one_tile) {
            const int t = tile - pre[li], tiles_x = (st.W + io.tox - 1) / io.tox;
            ty0 = (t / tiles_x) * io.toy;
            tx0 = (t % tiles_x) * io.tox;
        }
        q.W = st.W;
        q.We = st.We;
        q.c = st.c;
        q.P = st.P;
        q.ch = ch;
        q.psf_mode = io.psf_mode;
        q.scale = io.scale;
        q.hp = io.hperm + (long long)b * Kx * Ny;
        if (io.psf_mode) {
            q.in = io.psf + st.psf_off;
            q.hO = q.wO = 0;
            q.rows = Ny;
            q.width = Nx;
        } else {
            const long long at = (long long)ty0 * st.W + tx0;
            q.in = a.ext + ext_index(st, nchan, ch) + (long long)ty0 * st.We + tx0;
            q.out = a.y + y_index(st, nchan, ch) + at;
            q.hO = min(io.toy, st.H - ty0);
            q.wO = min(io.tox, st.W - tx0);
            q.rows = q.hO + 2 * st.c;
            q.width = q.wO + 2 * st.c;
            if (a.conv_chi2) {
                const Channel& chn = a.chan[(long long)b * a.chan_stride + ch];
                q.tmw = chn.mweight;
                q.tmsky = chn.msky;
                q.img = a.img + st.pix_off + at;
                q.sig = a.sig + st.pix_off + at;
                q.slot = st.wb_off + (long long)(ty0 / 16) * ((st.W + 31) / 32) + tx0 / 32;
            }
        }
        // row pairs come in groups of G (the last one may be smaller), each
        // exchanging through its own rows
        q.npair = (q.rows + 1) / 2;
        q.ngrp = (q.npair + SMALL_GROUP - 1) / SMALL_GROUP;
        q.G = (q.npair + q.ngrp - 1) / q.ngrp;
        const int npo = (q.hO + 1) / 2;
        q.ngo = (npo + SMALL_GROUP - 1) / SMALL_GROUP;
        q.Go = q.ngo ? (npo + q.ngo - 1) / q.ngo : 0;
    };
    if (it0 < it1 && tid == NT - 1) fill(it0, info[0]);
    for (long long it = it0; it < it1; ++it) {
        __syncthreads();  // the previous item is done with the spectrum, this one's info is there
        const TileItem& I = info[(it - it0) & 1];
        if (it + 1 < it1 && tid == NT - 1) fill(it + 1, info[(it + 1 - it0) & 1]);
        Ph::rows_a(spec, twx, I);
        __syncthreads();
        Ph::rows_b(spec, I);
        __syncthreads();
        Ph::cols_a(spec, twy, I);
        __syncthreads();
        Ph::cols_b(spec, I);
        if (io.psf_mode) continue;
        __syncthreads();
        Ph::cols_ai(spec, twy, I);
        __syncthreads();
        // output rows.  In an LM trial pass (a.conv_chi2) nothing is written: each
        // row pair's chi^2 per 32 columns goes to part[pair][column block], and the
        // 16 x 32 blocks' sums to the stamp's partial slots.
        for (int g = 0; g < I.ngo; ++g) {
            const int np = min(I.Go, (I.hO + 1) / 2 - g * I.Go);
            float2* area = spec + (I.c + 2 * g * I.Go) * Kx;
            Ph::out_b(area, I, g, np);
            __syncthreads();
            Ph::out_a(area, twx, I, g, np, a.conv_chi2);
            if (!a.conv_chi2) continue;
            __syncthreads();
            Ph::out_chi2(area, part, I, g, np);
        }
        if (a.conv_chi2) {
            // each 16 x 32 block: its 8 row pairs' partials merged in row order
            __syncthreads();
            const int nby = (I.hO + 15) / 16, nbw = (I.W + 31) / 32, nbx = (I.wO + 31) / 32, npo = (I.hO + 1) / 2;
            for (int q = tid; q < nby * nbx; q += NT) {
                const int by = q / nbx, bx = q - by * nbx;
                CSum cs = part[(8 * by) * nbx + bx];
                for (int pr = 8 * by + 1; pr < min(npo, 8 * by + 8); ++pr)
                    cs = csum_merge(cs, part[pr * nbx + bx]);
                a.partial[(I.slot + (long long)by * nbw + bx) * nchan + I.ch] = cs.s + cs.c;
            }
        }
        if (a.work && tid == 0) atomicAdd(&a.work[PROF_CONV], (unsigned long long)io.flops);
    }
}

template <int MX, int MY>
cudaError_t launch_small_t(const SmallIO& io, const PassArgs& a, const FFTArgs& f, long long items,
                           cudaStream_t s)
{
    static int optin[64];
    const size_t smem = small_smem(MX, MY);
    cudaError_t e = ensure_smem_optin((const void*)k_conv_fft_small<MX, MY>, (int)smem, optin);
    if (e != cudaSuccess) return e;
    const int grid = (int)std::min<long long>(items, 152LL * small_ctas_per_sm<MX, MY>());
    GF_LAUNCH_PDL(k_conv_fft_small<MX, MY>, dim3(grid), dim3(small_threads(MX)), smem, s, io, a,
                  (const float2*)f.tw_x, (const float2*)f.tw_y);
    GF_COUNT_LAUNCH();
    return cudaSuccess;
}

cudaError_t launch_small(const SmallIO& io, const PassArgs& a, const FFTArgs& f, long long items,
                         cudaStream_t s)
{
    switch (f.Nx * 256 + f.Ny) {
#define SMALL_CASE(NX_, NY_) \
    case NX_ * 256 + NY_: return launch_small_t<NX_ / 8, NY_ / 8>(io, a, f, items, s);
        SMALL_CASE(96, 96) SMALL_CASE(96, 128) SMALL_CASE(96, 160)
        SMALL_CASE(128, 96) SMALL_CASE(128, 128) SMALL_CASE(128, 160)
        SMALL_CASE(160, 96) SMALL_CASE(160, 128) SMALL_CASE(160, 160)
#undef SMALL_CASE
    default: return cudaErrorInvalidValue;
    }
}

size_t warp_row_smem(int N) { return sizeof(float2) * ((size_t)warp_fft_table_len(N) + (size_t)WROW_WARPS * N); }

// the warp row kernels exist for these Nx
#define WARP_FFT_CASES(X) X(3) X(4) X(5) X(6) X(8) X(9) X(10) X(12) X(15) X(16) X(18) X(20)

bool warp_rows_ok(int Nx)
{
    if (Nx % 32 != 0) return false;
    switch (Nx / 32) {
#define WF_CASE(M_) case M_:
        WARP_FFT_CASES(WF_CASE)
#undef WF_CASE
        return true;
    default: return false;
    }
}

}  // namespace

size_t fft_row_smem(int Nx) { return sizeof(float2) * 3 * (size_t)Nx; }

int fft_small_len(int n)
{
    for (int M = 3; M <= 5; ++M)
        if (32 * M >= n) return 32 * M;
    return 0;
}
size_t fft_col_smem(int Ny, int cpc) { return sizeof(float2) * ((size_t)2 * Ny * cpc + Ny); }

cudaError_t launch_fft_twiddles(const FFTArgs& f, cudaStream_t s)
{
    k_twiddles<<<(f.Nx + 255) / 256, 256, 0, s>>>(f.Nx, f.tw_x);
    GF_COUNT_LAUNCH();
    k_twiddles<<<(f.Ny + 255) / 256, 256, 0, s>>>(f.Ny, f.tw_y);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

static cudaError_t optin_all(const FFTArgs& f)
{
    static int o1[64], o2[64], o3[64];
    cudaError_t e = ensure_smem_optin((const void*)k_fft_rows_fwd, (int)fft_row_smem(f.Nx), o1);
    if (e == cudaSuccess)
        e = ensure_smem_optin((const void*)k_fft_rows_inv, (int)fft_row_smem(f.Nx), o2);
    if (e == cudaSuccess)
        e = ensure_smem_optin((const void*)k_fft_cols, (int)fft_col_smem(f.Ny, f.cpc), o3);
    return e;
}

// forward / inverse row pass over `pairs` row pairs of each of nprob problems:
// the warp kernels where Nx allows, else the shared-memory Stockham kernels
// a one-dimensional grid of nblk CTAs for each of nprob problems
static bool grid_ok(long long nblk, long long nprob) { return nblk * nprob <= 0x7fffffffLL; }

static cudaError_t rows_fwd(const FFTArgs& f, RowIO r, const PassArgs& a, int pairs,
                            int nprob, cudaStream_t s)
{
    if (warp_rows_ok(f.Nx)) {
        r.nblk = (pairs + WROW_WARPS - 1) / WROW_WARPS;
        if (!grid_ok(r.nblk, nprob)) return cudaErrorInvalidConfiguration;
        const dim3 grid((unsigned)((long long)r.nblk * nprob));
        switch (f.Nx / 32) {
#define WF_CASE(M_)                                                                          \
    case M_:                                                                                 \
        GF_LAUNCH_PDL(k_fft_rows_fwd_w<M_>, grid, dim3(WROW_WARPS * 32), warp_row_smem(f.Nx), \
                      s, f, r, a);                                                           \
        break;
            WARP_FFT_CASES(WF_CASE)
#undef WF_CASE
        default: return cudaErrorInvalidValue;
        }
    } else {
        r.nblk = pairs;
        if (!grid_ok(r.nblk, nprob)) return cudaErrorInvalidConfiguration;
        GF_LAUNCH_PDL(k_fft_rows_fwd, dim3((unsigned)((long long)pairs * nprob)), dim3(ROW_THREADS),
                      fft_row_smem(f.Nx), s, f, r, a);
    }
    GF_COUNT_LAUNCH();
    return cudaSuccess;
}

// column pass (mode 1: transform, PSF product, inverse; mode 0: forward only)
static cudaError_t cols_pass(const FFTArgs& f, ColIO c, const PassArgs& a, int nprob,
                             int mode, cudaStream_t s)
{
    const int Kx = f.Nx / 2 + 1;
    // fewer columns per CTA until the pass has four CTAs per SM (the column
    // pass waits on L2 loads: more, smaller CTAs keep more of them in flight)
    FFTArgs fc = f;
    if (mode == 1)
        while (fc.cpc > 2 && (long long)nprob * ((Kx + fc.cpc - 1) / fc.cpc) < 4 * 152) fc.cpc /= 2;
    fc.flops_col = f.flops_col * (float)fc.cpc / (float)f.cpc;
    c.nblk = (Kx + fc.cpc - 1) / fc.cpc;
    if (!grid_ok(c.nblk, nprob)) return cudaErrorInvalidConfiguration;
    GF_LAUNCH_PDL(k_fft_cols, dim3((unsigned)((long long)c.nblk * nprob)), dim3(COL_THREADS),
                  fft_col_smem(fc.Ny, fc.cpc), s, fc, c, a, mode);
    GF_COUNT_LAUNCH();
    return cudaSuccess;
}

static cudaError_t rows_inv(const FFTArgs& f, RowInvIO v, const PassArgs& a, int pairs,
                            int nprob, cudaStream_t s)
{
    if (warp_rows_ok(f.Nx)) {
        v.nblk = (pairs + WROW_WARPS - 1) / WROW_WARPS;
        if (!grid_ok(v.nblk, nprob)) return cudaErrorInvalidConfiguration;
        const dim3 grid((unsigned)((long long)v.nblk * nprob));
        switch (f.Nx / 32) {
#define WF_CASE(M_)                                                                          \
    case M_:                                                                                 \
        GF_LAUNCH_PDL(k_fft_rows_inv_w<M_>, grid, dim3(WROW_WARPS * 32), warp_row_smem(f.Nx), \
                      s, f, v, a);                                                           \
        break;
            WARP_FFT_CASES(WF_CASE)
#undef WF_CASE
        default: return cudaErrorInvalidValue;
        }
    } else {
        v.nblk = pairs;
        if (!grid_ok(v.nblk, nprob)) return cudaErrorInvalidConfiguration;
        GF_LAUNCH_PDL(k_fft_rows_inv, dim3((unsigned)((long long)pairs * nprob)), dim3(ROW_THREADS),
                      fft_row_smem(f.Nx), s, f, v, a);
    }
    GF_COUNT_LAUNCH();
    return cudaSuccess;
}

cudaError_t launch_psf_wrap(const FFTArgs& f, int count, const StampInfo* st, const float* psf,
                            cudaStream_t s)
{
    k_psf_wrap<<<dim3(8 * count), 256, 0, s>>>(f, count, st, psf);
    GF_COUNT_LAUNCH();
    return cudaGetLastError();
}

// PSF spectra of all stamps of a call (uniform size): wrap, row pass over all
// Ny rows, forward column pass.
cudaError_t launch_fft_psf(const FFTArgs& f, int count, const StampInfo* st, const float* psf,
                           cudaStream_t s)
{
    PassArgs none;
    memset(&none, 0, sizeof(none));
    if (f.small) {
        SmallIO io;
        memset(&io, 0, sizeof(io));
        io.one_tile = 1;
        io.st = st;
        io.psf = psf;
        io.scale = (float)(0.25 / ((double)f.Ny * (double)f.Nx));  // (see the unpacking)
        io.hperm = f.hhat;
        io.count = count;
        io.psf_mode = 1;
        const cudaError_t e = launch_small(io, none, f, count, s);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    cudaError_t e = optin_all(f);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(f.psfgrid, 0, sizeof(float) * (size_t)count * f.Ny * f.Nx, s);
    if (e != cudaSuccess) return e;
    k_psf_wrap<<<dim3(8 * count), 256, 0, s>>>(f, count, st, psf);
    GF_COUNT_LAUNCH();
    const int Kx = f.Nx / 2 + 1;
    RowIO r;
    r.in = f.psfgrid;
    r.in_stride = (long long)f.Ny * f.Nx;
    r.ld = f.Nx;
    r.width = f.Nx;
    r.rows = f.Ny;
    r.spec = f.hhat;
    r.spec_stride = (long long)f.Ny * Kx;
    r.out_rows = f.Ny;
    r.nchan = 1;
    e = rows_fwd(f, r, none, (f.Ny + 1) / 2, count, s);
    if (e != cudaSuccess) return e;
    ColIO c;
    c.spec = f.hhat;
    c.spec_stride = (long long)f.Ny * Kx;
    c.rows_in = f.Ny;
    c.row0 = 0;
    c.nrows_out = f.Ny;
    c.nchan = 1;
    e = cols_pass(f, c, none, count, 0, s);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// Convolve the pass's channel grids (a.ext) into a.y through the spectrum
// scratch `spec` (count * nchan * He * Kx complex values).
cudaError_t launch_conv_fft(const PassArgs& a, const FFTArgs& f, float2* spec, cudaStream_t s)
{
    const StampInfo& s0 = f.st0;  // uniform stamp geometry (host copy)
    const int Kx = f.Nx / 2 + 1;
    if (f.small) {
        SmallIO io;
        memset(&io, 0, sizeof(io));
        io.toy = f.toy;
        io.tox = f.tox;
        io.one_tile = f.one_tile;
        io.st = a.st;
        io.hperm = f.hhat;
        const int He = f.toy + 2 * s0.c;
        io.flops = (float)(((He + 1) / 2 + (f.toy + 1) / 2) * 5.0 * f.Nx * log2((double)f.Nx) +
                           Kx * (10.0 * f.Ny * log2((double)f.Ny) + 6.0 * f.Ny));
        const cudaError_t e = launch_small(io, a, f, a.maxitems[WK_CONV], s);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    const int nprob = a.count * a.nchan;
    cudaError_t e = optin_all(f);
    if (e != cudaSuccess) return e;
    RowIO r;
    r.in = a.ext;
    r.in_stride = (long long)s0.He * s0.We;
    r.ld = s0.We;
    r.width = s0.We;
    r.rows = s0.He;
    r.spec = spec;
    r.spec_stride = (long long)s0.He * Kx;
    r.out_rows = s0.He;
    r.nchan = a.nchan;
    e = rows_fwd(f, r, a, (s0.He + 1) / 2, nprob, s);
    if (e != cudaSuccess) return e;
    ColIO c;
    c.spec = spec;
    c.spec_stride = (long long)s0.He * Kx;
    c.rows_in = s0.He;
    c.row0 = s0.c;
    c.nrows_out = s0.H;
    c.nchan = a.nchan;
    e = cols_pass(f, c, a, nprob, 1, s);
    if (e != cudaSuccess) return e;
    RowInvIO v;
    v.spec = spec;
    v.spec_stride = (long long)s0.He * Kx;
    v.row0 = s0.c;
    v.col0 = s0.c;
    v.H = s0.H;
    v.W = s0.W;
    v.out = a.y;
    v.out_stride = (long long)s0.H * s0.W;
    v.nchan = a.nchan;
    e = rows_inv(f, v, a, (s0.H + 1) / 2, nprob, s);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// Image preparation, model projection and PSF application (sm_103a).
//
//   k_prepare_images  per image: float64 moments C_o, C_oo (Sec. 3: precomputed image constants),
//                     zero-mean real-to-half-complex transform (Sec. 3.3: the observed images'
//                     transforms are precomputed once), unit-norm spectrum (C_oo by Plancherel).
//   k_project         per orientation: rotate the atoms by the quaternion (Sec. 3.1) and integrate
//                     each Gaussian atom over z and over every pixel (Eq. 1) into I0.
//   k_ctf_table       per PSF grid point: CTF(s) Env(s) on the half-spectrum grid (Eq. 4's forms).
//   k_psf_spectra     per orientation: transform I0, multiply by each PSF (Eq. 5), float64 moment
//                     B = n C_cc - C_c^2 (Plancherel), unit-norm spectrum per parameter set.
//   k_psf_real        the synthetic map I1 = F^-1[F(I0) CTF Env] in real space (Sec. 3.8).
//
// The forward transforms here use exp(-2 pi i k x / N).  For a real image this is the complex
// conjugate of Eq. 2's transform; the scoring kernel applies the matching inverse phase, so the
// correlation it evaluates is C_co(d) = sum_r o(r) I1(r + d) with d as in Eq. 7.  These
// transforms run once per image and once per orientation, so they are plain dense DFT sums over
// shared memory, but for the maps', which go by factors; the hot loop is the scoring kernel.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>

#include "bioem_internal.cuh"

namespace {

// Threads of the transform kernels: two blocks per SM up to 128 px; at 192 px a block's spectrum fills
// the SM's shared memory, so it has 512.
template <int N>
struct Dft {
    static constexpr int T = N == 192 ? 512 : 256;
    static constexpr int NC = N / 2, H = NC + 1;
    // Register tiles: 16 lanes share a group's KY rows (or frequencies) and take KX columns each, 16
    // apart.  A dense sum costs N multiply-adds per output either way; the tile is what lets a value
    // loaded from shared memory serve 8 (x KX) or 4 (x KY) of them at 128 px instead of one.
    static constexpr int G = T / 16, KY = N / G, KX = NC / 16;
    static_assert(KY * G == N && KX * 16 == NC, "whole tiles; the kx = N/2 column is summed apart");
    static constexpr int PER = (N * H + T - 1) / T;   // coefficients per thread in the passes over a spectrum
};

// Deterministic block sums of two doubles (fixed order: lanes, then warps); red holds 2 T / 32 doubles.
template <int T>
__device__ __forceinline__ void block_sum2(double& a, double& b, double* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, off);
        b += __shfl_xor_sync(0xffffffffu, b, off);
    }
    if (lane == 0) {
        red[warp] = a;
        red[T / 32 + warp] = b;
    }
    __syncthreads();
    a = red[0];
    b = red[T / 32];
    for (int w = 1; w < T / 32; ++w) {
        a += red[w];
        b += red[T / 32 + w];
    }
    __syncthreads();
}

// Largest value over the block, in every thread; red holds T / 32 floats.
template <int T>
__device__ __forceinline__ float block_max(float v, float* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
    if (lane == 0) red[warp] = v;
    __syncthreads();
    v = red[0];
    for (int w = 1; w < T / 32; ++w) v = fmaxf(v, red[w]);
    __syncthreads();
    return v;
}

// (idx + step) mod N for idx, step < N: the smaller of the two candidates as unsigned numbers
template <int N>
__device__ __forceinline__ unsigned step_mod(unsigned idx, unsigned step) {
    if constexpr ((N & (N - 1)) == 0) return (idx + step) & (N - 1);
    else return min(idx + step, idx + step - N);
}

// Shared memory of the transform kernels.
template <int N>
struct DftSm {
    float2* F;      // [N][H]
    float2* tw;     // [N] exp(-2 pi i t / N)
    float2* ts;     // [N] the same with its parts exchanged: (w.y, w.x)
    double* red;    // [4 T / 32]
    __device__ __forceinline__ explicit DftSm(unsigned char* smem) {
        F = reinterpret_cast<float2*>(smem);
        tw = F + N * Dft<N>::H;
        ts = tw + N;
        red = reinterpret_cast<double*>(ts + N);
    }
    // the twiddle pair of the forward transform, or of the inverse (conjugates)
    __device__ __forceinline__ void twiddles(const float2* __restrict__ g_tw, bool inverse) const {
        for (int i = threadIdx.x; i < N; i += Dft<N>::T) {
            const float2 w = g_tw[i];
            const float y = inverse ? -w.y : w.y;
            tw[i] = make_float2(w.x, y);
            ts[i] = make_float2(y, w.x);
        }
    }
    static constexpr size_t bytes() {
        return (size_t)(N * Dft<N>::H + 2 * N) * sizeof(float2) + 4 * (Dft<N>::T / 32) * sizeof(double);
    }
};

// F[y][kx] = sum_x (img[y][x] - mean) W^(kx x), kx = 0..N/2 (row pass of a real 2-D transform), x ascending
// in one FP32 accumulator per output.
template <int N, bool VEC = true>
__device__ __forceinline__ void r2c_rows(const float* __restrict__ img, float mean, const DftSm<N>& sm) {
    // four pixels of a row; VEC: img is 16-byte aligned
    auto load4 = [](const float* p) {
        if constexpr (VEC) return __ldg(reinterpret_cast<const float4*>(p));
        else return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
    };
    using D = Dft<N>;
    constexpr int H = D::H, KY = D::KY, KX = D::KX;
    const int g = threadIdx.x >> 4, l = threadIdx.x & 15;
    float2 acc[KY][KX];
    unsigned idx[KX];
#pragma unroll
    for (int k = 0; k < KX; ++k) {
        idx[k] = 0;
#pragma unroll
        for (int i = 0; i < KY; ++i) acc[i][k] = make_float2(0.f, 0.f);
    }
#pragma unroll 1
    for (int x0 = 0; x0 < N; x0 += 4) {
        float v[KY][4];
#pragma unroll
        for (int i = 0; i < KY; ++i) {
            const float4 q = load4(img + (size_t)(g * KY + i) * N + x0);
            v[i][0] = q.x - mean; v[i][1] = q.y - mean; v[i][2] = q.z - mean; v[i][3] = q.w - mean;
        }
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int k = 0; k < KX; ++k) {
                const float2 w = sm.tw[idx[k]];
                idx[k] = step_mod<N>(idx[k], l + 16 * k);
#pragma unroll
                for (int i = 0; i < KY; ++i) acc[i][k] = __ffma2_rn(make_float2(v[i][x], v[i][x]), w, acc[i][k]);
            }
    }
#pragma unroll
    for (int i = 0; i < KY; ++i)
#pragma unroll
        for (int k = 0; k < KX; ++k) sm.F[(g * KY + i) * H + l + 16 * k] = acc[i][k];
    if (threadIdx.x < N) {   // kx = N/2: the twiddles alternate between t = 0 and N/2
        const float* row = img + (size_t)threadIdx.x * N;
        float2 a = make_float2(0.f, 0.f);
        const float2 w0 = sm.tw[0], w1 = sm.tw[N / 2];
        for (int x0 = 0; x0 < N; x0 += 4) {
            const float4 q = load4(row + x0);
            const float v[4] = {q.x - mean, q.y - mean, q.z - mean, q.w - mean};
#pragma unroll
            for (int x = 0; x < 4; ++x) a = __ffma2_rn(make_float2(v[x], v[x]), (x & 1) ? w1 : w0, a);
        }
        sm.F[threadIdx.x * H + N / 2] = a;
    }
}

// In place over shared memory: F[ky][kx] <- sum_y F[y][kx] W^(ky y) with the twiddles in sm.tw (column
// pass; the inverse with conjugate twiddles), y ascending, re and im each in one FP32 accumulator.  All
// outputs are held in registers until every read is done.
template <int N>
__device__ __forceinline__ void c2c_columns_inplace(const DftSm<N>& sm) {
    using D = Dft<N>;
    constexpr int H = D::H, KY = D::KY, KX = D::KX;
    const int g = threadIdx.x >> 4, l = threadIdx.x & 15;
    float2 acc[KY][KX];
    unsigned idx[KY];
#pragma unroll
    for (int i = 0; i < KY; ++i) {
        idx[i] = 0;
#pragma unroll
        for (int k = 0; k < KX; ++k) acc[i][k] = make_float2(0.f, 0.f);
    }
#pragma unroll 2
    for (int y = 0; y < N; ++y) {
        float2 v[KX];
#pragma unroll
        for (int k = 0; k < KX; ++k) v[k] = sm.F[y * H + l + 16 * k];
#pragma unroll
        for (int i = 0; i < KY; ++i) {
            const float2 w = sm.tw[idx[i]], ws = sm.ts[idx[i]];
            idx[i] = step_mod<N>(idx[i], g * KY + i);
#pragma unroll
            for (int k = 0; k < KX; ++k) {
                // re += -v.y w.y, then v.x w.x; im += v.y w.x, then v.x w.y
                acc[i][k] = __ffma2_rn(make_float2(-v[k].y, v[k].y), ws, acc[i][k]);
                acc[i][k] = __ffma2_rn(make_float2(v[k].x, v[k].x), w, acc[i][k]);
            }
        }
    }
    float2 last = make_float2(0.f, 0.f);   // kx = N/2, one ky per thread
    if (threadIdx.x < N) {
        unsigned t = 0;
        for (int y = 0; y < N; ++y) {
            const float2 v = sm.F[y * H + N / 2];
            const float2 w = sm.tw[t], ws = sm.ts[t];
            t = step_mod<N>(t, threadIdx.x);
            last = __ffma2_rn(make_float2(-v.y, v.y), ws, last);
            last = __ffma2_rn(make_float2(v.x, v.x), w, last);
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < KY; ++i)
#pragma unroll
        for (int k = 0; k < KX; ++k) sm.F[(g * KY + i) * H + l + 16 * k] = acc[i][k];
    if (threadIdx.x < N) sm.F[threadIdx.x * H + N / 2] = last;
    __syncthreads();
}

// The inverse row pass: real[y][x] = G(0) + (-1)^x G(N/2) + 2 sum_{0 < kx < N/2} Re(G(kx) exp(+2 pi i kx x / N)) of the
// rows G of sm.F, kx ascending; put(y, x, value) for every pixel.  sm.tw holds the FORWARD twiddles.
template <int N, class PUT>
__device__ __forceinline__ void c2r_rows(const DftSm<N>& sm, PUT&& put) {
    using D = Dft<N>;
    constexpr int H = D::H, KY = D::KY, KX = N / 16;
    const int g = threadIdx.x >> 4, l = threadIdx.x & 15;
    float acc[KY][KX];
    unsigned idx[KX];
#pragma unroll
    for (int k = 0; k < KX; ++k) {
        idx[k] = l + 16 * k;
#pragma unroll
        for (int i = 0; i < KY; ++i) acc[i][k] = 0.f;
    }
#pragma unroll 1
    for (int kx = 1; kx < N / 2; ++kx) {
        float2 v[KY];
#pragma unroll
        for (int i = 0; i < KY; ++i) v[i] = sm.F[(g * KY + i) * H + kx];
#pragma unroll
        for (int k = 0; k < KX; ++k) {
            const float2 w = sm.tw[idx[k]];   // exp(-2 pi i kx x / N); conjugated below
            idx[k] = step_mod<N>(idx[k], l + 16 * k);
#pragma unroll
            for (int i = 0; i < KY; ++i) acc[i][k] = fmaf(v[i].x, w.x, fmaf(v[i].y, w.y, acc[i][k]));
        }
    }
#pragma unroll
    for (int i = 0; i < KY; ++i) {
        const int y = g * KY + i;
        const float g0 = sm.F[y * H].x, gn = sm.F[y * H + N / 2].x;
#pragma unroll
        for (int k = 0; k < KX; ++k) {
            const int x = l + 16 * k;
            const float v = g0 + ((x & 1) ? -gn : gn);
            put(y, x, v + 2.f * acc[i][k]);
        }
    }
}

// Write F * T * scale (T may be null; DC zeroed) to a [N][N/2 + 1] half spectrum; returns the calling thread's
// largest |coefficient|.
template <int N>
__device__ __forceinline__ float store_half_spectrum(const float2* F, const float* __restrict__ T, float scale,
                                                     float2* __restrict__ spec) {
    float amax = 0.f;
    for (int o = threadIdx.x; o < N * Dft<N>::H; o += Dft<N>::T) {
        float2 v = F[o];
        if (T) v = c_scale(v, __ldg(T + o));
        v = c_scale(v, scale);
        if (o == 0) v = make_float2(0.f, 0.f);
        spec[o] = v;
        amax = fmaxf(amax, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    return amax;
}

// w_kx |v|^2 of coefficient o of the half spectrum, w_kx = 1 on the kx = 0 and kx = N/2 columns and 2 elsewhere
// (their Hermitian partners).  DC is left out, not multiplied by 0: it alone may be infinite (the sum of an
// image whose other coefficients are within range).
template <int N>
__device__ __forceinline__ double half_energy(int o, float2 v) {
    const int kx = o % Dft<N>::H;
    const double m = (double)v.x * v.x + (double)v.y * v.y;
    return o == 0 ? 0.0 : (kx == 0 || kx == N / 2) ? m : 2.0 * m;
}

// VEC: the images start on a 16-byte boundary (a caller's tensor may be a view that does not).
template <int N, bool VEC>
__global__ void __launch_bounds__(Dft<N>::T) k_prepare_images(const float* __restrict__ images,
                                                              const float2* __restrict__ g_tw,
                                                              float2* __restrict__ spec,
                                                              double* __restrict__ kA, float* __restrict__ amax,
                                                              double cn,
                                                              int* __restrict__ status) {
    constexpr int H = Dft<N>::H, T = Dft<N>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    const DftSm<N> sm(smem);
    const int w = blockIdx.x;
    const float* img = images + (size_t)w * N * N;
    sm.twiddles(g_tw, false);

    double s1 = 0.0, s2 = 0.0;
    for (int i = threadIdx.x; i < N * N; i += T) {
        const double v = img[i];
        s1 += v;
        s2 += v * v;
    }
    block_sum2<T>(s1, s2, sm.red);
    const double n = (double)N * N;
    const double A = n * s2 - s1 * s1;   // n C_oo - C_o^2
    const float mean = (float)(s1 / n);

    r2c_rows<N, VEC>(img, mean, sm);
    __syncthreads();
    c2c_columns_inplace<N>(sm);
    double e = 0.0, dummy = 0.0;
    for (int o = threadIdx.x; o < N * H; o += T) e += half_energy<N>(o, sm.F[o]);
    block_sum2<T>(e, dummy, sm.red);
    const bool bad = !(A > 0.0) || !(e > 0.0);
    const float scale = bad ? 0.f : (float)(1.0 / sqrt(e));
    const float mx = block_max<T>(store_half_spectrum<N>(sm.F, nullptr, scale, spec + (size_t)w * N * H),
                                  reinterpret_cast<float*>(sm.red));
    if (threadIdx.x == 0) {
        amax[w] = mx;
        if (bad) {
            atomicOr(status, BIOEM_DEV_NUMERIC);
            kA[w] = -INFINITY;
        } else {
            kA[w] = 0.5 * (3.0 - n) * log(A) + cn;
        }
    }
}

// Pixel integral of a unit Gaussian between two boundaries whose scaled positions are a0 < a1,
// given T = erfc(|a|) and the sign of a at each boundary; written without cancellation in either
// tail: for a0, a1 > 0 it is (T0 - T1) / 2, for a0, a1 < 0 it is (T1 - T0) / 2.
__device__ __forceinline__ float pixel_mass(float t0, bool neg0, float t1, bool neg1) {
    if (!neg0) return 0.5f * (t0 - t1);
    if (neg1) return 0.5f * (t1 - t0);
    return 0.5f * ((1.f - t0) + (1.f - t1));
}

// |u| beyond which erfc(|u|) (about 1.4e-54 at 11) is zero in FP32: boundaries past it are taken as zero
// without evaluating erfc.  An atom's window of pixels reaches to |u| = kWindow: past it both boundaries
// of a pixel give zero already (erfc(10.4) < 1e-48, below half the smallest FP32 number), so the pixel
// integral is exactly zero, with room for the rounding of the window's own bounds.
constexpr float kErfcZero = 11.f, kWindow = 10.5f;

// k_project's reach: kWindow, but one pixel (D) more for atoms that are points beside a pixel.  The bounds of a
// window are rounded by up to 5e-5 pixels (N 2^-22), for which kWindow leaves 0.4 / D.  (Formed in the kernel,
// in a register or in shared memory, it cost 3 % of 1024 maps at 128 px.)
float window_reach(double sigma, double pixel) {
    const double d = pixel / (sigma * 1.4142135623730951);
    return d > 4096.0 ? (float)(kWindow + d) : kWindow;
}

// One orientation per block.  The image is cut into tiles of TR x TC pixels, LR x LC per lane (4 x 8 lanes);
// a warp owns TPW tiles, one in each of TPW bands of rows and in different columns, so that dense and
// empty parts of the projection even out.  Atoms are processed in chunks of 32 in order: a warp tabulates
// the pixel integrals of its share of the next chunk's atoms over their windows only (a half warp per axis,
// 15 pixels per pass), then each warp goes through the atoms whose window meets its tile (one ballot per
// tile and chunk) and accumulates w_a gy gx as packed FP32 pairs.  Every pixel sums its atoms in index
// order; left out are exact zeros only.  A chunk's positions are formed (float64, one warp, lane = atom) two
// chunks ahead of its sums and its tables one chunk ahead: one barrier per chunk.
// Bound by issue (0.7 per cycle and scheduler) and the latency of erfc: ~540 warp instructions per atom at 128 px
// (1.1 A), most of them for the tables' three passes and for 6.7 tiles' sums.  128 px, 5000 atoms, sigma 1.5 A, us per orientation: 7.1 when every boundary
// of the image was tabulated for every atom and whole rows were summed, 3.4 with 8 warps of 4 tiles, 3.1
// with 16 warps of 2, 2.7 with atoms taken by the warps that are free.
template <int N>
struct ProjCfg {
    static constexpr int LR = N == 32 ? 2 : 4, LC = LR;
    static constexpr int TR = 4 * LR, TC = 8 * LC;                 // tile
    static constexpr int TCOLS = N / TC, TROWS = N / TR;
    static constexpr int NW = N == 96 ? 18 : N == 128 ? 16 : N == 192 ? 24 : 8;   // warps
    static constexpr int BAND = NW / TCOLS, TPW = TROWS / BAND;    // tile rows per band, tiles per warp
    static_assert(TCOLS * TC == N && TROWS * TR == N && BAND * TCOLS == NW && TPW * BAND == TROWS, "tiles cover the image");
    static constexpr int T = 32 * NW;
    // Warps take the atoms they tabulate one by one, after their sums, so that those with sparse tiles tabulate
    // more: 1024 maps at 128 px 3.07 -> 2.78 ms, 500 at 192 px 5.59 -> 3.03 ms.  At 96 px (two passes per
    // atom) and below equal shares are as good or better: 1000 maps 2.46 against 2.45 ms, at 64 px 1.51 against 1.61.
    static constexpr bool TAKE = N >= 128;
    static constexpr int CH = 32;                                  // atoms per chunk: one per lane of a ballot
    static constexpr size_t SM_TAB = (size_t)CH * 2 * N * sizeof(float);   // gx, gy rows of a chunk
    static constexpr size_t SMEM = 2 * SM_TAB;
};

template <int V>
__device__ __forceinline__ void load_vec(const float* src, float (&v)[V]) {
    if constexpr (V == 4) {
        const float4 t = *reinterpret_cast<const float4*>(src);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
        const float2 t = *reinterpret_cast<const float2*>(src);
        v[0] = t.x; v[1] = t.y;
    }
}

template <int N>
__global__ void __launch_bounds__(ProjCfg<N>::T, N <= 64 ? 4 : N <= 128 ? 2 : 1) k_project(const float4* __restrict__ atoms, int n_atoms,
                                                           const float4* __restrict__ quats, double sigma,
                                                           double pixel, float reach, float* __restrict__ out) {
    using C = ProjCfg<N>;
    constexpr int LR = C::LR, LC = C::LC, CH = C::CH, NW = C::NW;
    extern __shared__ __align__(16) float tab[];   // [2][CH][2][N]: gx, gy (gy carries the atom's weight)
    __shared__ double rot[6];
    // per atom and axis, u_j = (edge_j - a) / (sigma sqrt 2) = j D - A as float pairs (hi + lo), so the tables run
    // in FP32 (an FMA forms j D_hi - A_hi exactly before rounding) with the accuracy of a float64
    // evaluation of u rounded to float; and the window [lo, hi] of pixels (empty where the chunk has no atom)
    struct Axis { float h, l; int lo, hi; };
    __shared__ Axis pos[3][CH][2];
    __shared__ float wgt[3][CH];
    __shared__ int taken[2];   // atoms of table 0 / 1's chunk that warps have taken

    const int q = blockIdx.x;
    if (threadIdx.x == 0) {
        const float4 qq = quats[q];
        double w = qq.x, x = qq.y, y = qq.z, z = qq.w;
        const double nrm = sqrt(w * w + x * x + y * y + z * z);
        w /= nrm; x /= nrm; y /= nrm; z /= nrm;
        rot[0] = 1.0 - 2.0 * (y * y + z * z); rot[1] = 2.0 * (x * y - w * z); rot[2] = 2.0 * (x * z + w * y);
        rot[3] = 2.0 * (x * y + w * z); rot[4] = 1.0 - 2.0 * (x * x + z * z); rot[5] = 2.0 * (y * z - w * x);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double inv = 1.0 / (sigma * 1.4142135623730951);
    const double dd = pixel * inv;                 // D: the pixel in units of sigma sqrt 2
    const float d_hi = (float)dd, d_lo = (float)(dd - (double)d_hi);
    const float inv_d = (float)(1.0 / dd);
    const double a_off = (0.5 * N + 0.5) * pixel;  // edge_j = j pixel - a_off

    auto positions = [&](int a0, int buf) {   // one warp: the chunk's positions and windows
        const int a = a0 + lane;
        Axis ax{0.f, 0.f, 0, -1}, ay{0.f, 0.f, 0, -1};
        float w = 0.f;
        if (a < n_atoms) {
            const float4 p = atoms[a];
            const double x = ((rot[0] * p.x + rot[1] * p.y + rot[2] * p.z) + a_off) * inv;
            const double y = ((rot[3] * p.x + rot[4] * p.y + rot[5] * p.z) + a_off) * inv;
            ax.h = (float)x; ax.l = (float)(x - (double)ax.h);
            ay.h = (float)y; ay.l = (float)(y - (double)ay.h);
            w = p.w;
            // boundary j has |u_j| < reach for (A - reach) / D < j < (A + reach) / D; pixel j has boundaries j, j + 1
            auto window = [&](Axis& v) {
                v.lo = max(0, (int)ceilf(fminf(fmaxf((v.h - reach) * inv_d, -1.e6f), 1.e6f)) - 1);
                v.hi = min(N - 1, (int)floorf(fminf(fmaxf((v.h + reach) * inv_d, -1.e6f), 1.e6f)));
            };
            window(ax);
            window(ay);
            if (!(fabsf(w) < INFINITY)) {
                // inf or NaN times the zeros beside the window is NaN: the whole image for an atom whose rows
                // come near it, so that the projection is found degenerate
                const bool near_rows = floorf((ay.h - kErfcZero) * inv_d) - 2.f < N && ceilf((ay.h + kErfcZero) * inv_d) + 1.f >= 0.f;
                ax.lo = ay.lo = 0;
                ax.hi = ay.hi = near_rows ? N - 1 : -1;
            }
        }
        pos[buf][lane][0] = ax;
        pos[buf][lane][1] = ay;
        wgt[buf][lane] = w;
    };
    auto tables = [&](int pb, int buf) {   // every warp: its share of the chunk in pos[pb], into table buf
        const int axis = lane >> 4, l = lane & 15;
        auto take = [&]() {
            int a = 0;
            if (lane == 0) a = atomicAdd(&taken[buf], 1);
            return __shfl_sync(0xffffffffu, a, 0);
        };
        for (int a = C::TAKE ? take() : warp; a < CH; a = C::TAKE ? take() : a + NW) {
            const Axis v = pos[pb][a][axis];
            const Axis o = pos[pb][a][axis ^ 1];
            if (v.hi < v.lo || o.hi < o.lo) continue;   // off the image on an axis (the same in both half warps)
            const float w = wgt[pb][a];
            float* both = tab + (size_t)(buf * CH + a) * 2 * N;
            float* row = both + axis * N;
            if constexpr (N == 32) {
                // a window is most of the image: a lane per pixel, both axes and boundaries at once, four erfc in flight
                // and no zeros to store (500 atoms, 1152 orientations, 2 PSFs, the whole call: 291 us with whole
                // rows summed, 324 with windows as below, 252 so)
                const Axis x = axis ? o : v, y = axis ? v : o;
                const float fj = (float)lane, fk = fj + 1.f;
                auto at = [&](const Axis& p, float j) { return fmaf(j, d_hi, -p.h) + fmaf(j, d_lo, -p.l); };
                const float x0 = at(x, fj), x1 = at(x, fk), y0 = at(y, fj), y1 = at(y, fk);
                const float ex0 = erfcf(fabsf(x0)), ex1 = erfcf(fabsf(x1)), ey0 = erfcf(fabsf(y0)), ey1 = erfcf(fabsf(y1));
                both[lane] = pixel_mass(ex0, x0 < 0.f, ex1, x1 < 0.f);
                both[N + lane] = w * pixel_mass(ey0, y0 < 0.f, ey1, y1 < 0.f);
                continue;
            }
            for (int i = 4 * lane; i < 2 * N; i += 128) *reinterpret_cast<float4*>(both + i) = make_float4(0.f, 0.f, 0.f, 0.f);
            __syncwarp();
            const int n = max(v.hi - v.lo, o.hi - o.lo) + 1;
            for (int b = 0; b < n; b += 15) {
                const int j = v.lo + b + l;
                const float fj = (float)j;
                const float u = fmaf(fj, d_hi, -v.h) + fmaf(fj, d_lo, -v.l);
                float t = 0.f;
                if (fabsf(u) < kErfcZero) t = erfcf(fabsf(u));
                const float t1 = __shfl_down_sync(0xffffffffu, t, 1);
                const float u1 = __shfl_down_sync(0xffffffffu, u, 1);
                const float m = pixel_mass(t, u < 0.f, t1, u1 < 0.f);
                if (l < 15 && j <= v.hi) row[j] = axis ? w * m : m;
            }
        }
    };

    float2 acc[C::TPW][LR / 2][LC];
#pragma unroll
    for (int t = 0; t < C::TPW; ++t)
#pragma unroll
        for (int i = 0; i < LR / 2; ++i)
#pragma unroll
            for (int j = 0; j < LC; ++j) acc[t][i][j] = make_float2(0.f, 0.f);
    const int lr = (lane >> 3) * LR, lc = (lane & 7) * LC;

    if (threadIdx.x < 2) taken[threadIdx.x] = 0;
    if (warp == 0) positions(0, 0);
    if (warp == NW - 1) positions(CH, 1);
    __syncthreads();
    tables(0, 0);
    __syncthreads();
    int pb = 0, buf = 0;   // this chunk's buffers: positions c mod 3, tables c mod 2
    for (int a0 = 0, c = 0; a0 < n_atoms; a0 += CH, ++c, buf ^= 1) {
        const int p1 = pb == 2 ? 0 : pb + 1, p2 = p1 == 2 ? 0 : p1 + 1;
        const Axis px = pos[pb][lane][0], py = pos[pb][lane][1];
        const bool some = px.lo <= px.hi && py.lo <= py.hi;
        if (warp == c % NW && a0 + 2 * CH < n_atoms) positions(a0 + 2 * CH, p2);
        if (!C::TAKE && a0 + CH < n_atoms) tables(p1, buf ^ 1);
        const float* base = tab + (size_t)buf * CH * 2 * N;
#pragma unroll
        for (int t = 0; t < C::TPW; ++t) {
            const int r0 = (warp / C::TCOLS + t * C::BAND) * C::TR, c0 = (warp + t) % C::TCOLS * C::TC;
            unsigned hit = __ballot_sync(0xffffffffu, some && px.lo < c0 + C::TC && px.hi >= c0 && py.lo < r0 + C::TR &&
                                                          py.hi >= r0);
            const float *tx = base + c0 + lc, *ty = base + N + r0 + lr;
            auto add = [&](int a) {
                float vx[LC], vy[LR];
                load_vec<LC>(tx + a * 2 * N, vx);
                load_vec<LR>(ty + a * 2 * N, vy);
#pragma unroll
                for (int i = 0; i < LR / 2; ++i)
#pragma unroll
                    for (int j = 0; j < LC; ++j)
                        acc[t][i][j] = __ffma2_rn(make_float2(vy[2 * i], vy[2 * i + 1]), make_float2(vx[j], vx[j]), acc[t][i][j]);
            };
            if constexpr (N == 32) {
                if (hit == 0xffffffffu) {   // nearly always: all of the chunk's atoms, loads ahead of the sums
#pragma unroll 16
                    for (int a = 0; a < CH; ++a) add(a);
                    hit = 0;
                }
            }
            while (hit) {
                const int a = __ffs(hit) - 1;
                hit &= hit - 1;
                add(a);
            }
        }
        if (C::TAKE && a0 + CH < n_atoms) tables(p1, buf ^ 1);
        if (threadIdx.x == 0) taken[buf] = 0;   // next taken from after the barrier
        pb = p1;
        __syncthreads();
    }
    float* o = out + (size_t)q * N * N;
#pragma unroll
    for (int t = 0; t < C::TPW; ++t) {
        const int r0 = (warp / C::TCOLS + t * C::BAND) * C::TR + lr, c0 = (warp + t) % C::TCOLS * C::TC + lc;
#pragma unroll
        for (int i = 0; i < LR; ++i) {
            float* row = o + (size_t)(r0 + i) * N + c0;
            float v[LC];
#pragma unroll
            for (int j = 0; j < LC; ++j) v[j] = (i & 1) ? acc[t][i / 2][j].y : acc[t][i / 2][j].x;
            if constexpr (LC == 4) *reinterpret_cast<float4*>(row) = make_float4(v[0], v[1], v[2], v[3]);
            else *reinterpret_cast<float2*>(row) = make_float2(v[0], v[1]);
        }
    }
}

// T[c][ky][kx] = CTF(s) Env(s) for PSF c on the half-spectrum grid, evaluated in float64.
// coef[4c..4c+3] = (a, A, b, sqrt(1 - A^2)); s = 2 pi (kx~, ky~) / (N pixel) with signed frequency
// indices.  The value depends on kx~^2 + ky~^2 only, so each unordered pair {|kx~|, |ky~|} is
// evaluated once and written to its (up to four) places: bound by float64 arithmetic, a quarter of
// evaluating every coefficient (1.20 ms for 1024 PSFs at 128 px before).
__global__ void k_ctf_table(const double* __restrict__ coef, int nctf, int N, double pixel,
                            float* __restrict__ T) {
    const int H = N / 2 + 1, tri = H * (H + 1) / 2;
    const long long total = (long long)nctf * tri;
    const double f = 2.0 * 3.14159265358979323846 / (N * pixel);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i / tri);
        const int r = (int)(i - (long long)c * tri);
        // r = hi (hi + 1) / 2 + lo, lo <= hi
        int hi = (int)((sqrtf(8.f * (float)r + 1.f) - 1.f) * 0.5f);
        while ((hi + 1) * (hi + 2) / 2 <= r) ++hi;
        while (hi * (hi + 1) / 2 > r) --hi;
        const int lo = r - hi * (hi + 1) / 2;
        const double s2 = f * f * ((double)lo * lo + (double)hi * hi);
        const double a = coef[4 * c], A = coef[4 * c + 1], b = coef[4 * c + 2];
        double sn, cs;
        sincos(0.5 * a * s2, &sn, &cs);
        const double ctf = -A * cs - coef[4 * c + 3] * sn;
        const float v = (float)(ctf * exp(-0.5 * b * s2));
        auto put = [&](int ky, int kx) { T[(size_t)c * N * H + (size_t)ky * H + kx] = v; };
        put(lo, hi);
        if (lo > 0 && lo < N / 2) put(N - lo, hi);
        if (lo != hi) {
            put(hi, lo);
            if (hi < N / 2) put(N - hi, lo);
        }
    }
}

// a + b and its rounding error (Knuth), two numbers side by side
__device__ __forceinline__ float2 two_sum(float2 a, float2 b, float2& err) {
    const float2 minus = make_float2(-1.f, -1.f);
    const float2 s = __fadd2_rn(a, b), t = __ffma2_rn(a, minus, s);
    err = __fadd2_rn(__ffma2_rn(__ffma2_rn(t, minus, s), minus, a), __ffma2_rn(t, minus, b));
    return s;
}

// hi + mid + lo += w v^2 for both parts of v, w a power of two: the square and the sums with their rounding errors
// (error-free transforms of Dekker and Knuth), to about 2^-66 of the sum for a spectrum's share of one thread.
__device__ __forceinline__ void add_square(float2& hi, float2& mid, float2& lo, float2 v, float2 w) {
    const float2 p = __fmul2_rn(v, v), e = __ffma2_rn(v, v, make_float2(-p.x, -p.y));
    float2 e1, e2, e3;
    hi = two_sum(hi, __fmul2_rn(p, w), e1);
    mid = two_sum(mid, e1, e2);
    mid = two_sum(mid, __fmul2_rn(e, w), e3);
    lo = __fadd2_rn(lo, __fadd2_rn(e2, e3));
}

// The sum of both parts, rounded to float64 (the two of hi and of mid are added exactly in FP32: each conversion to
// float64 and each float64 sum takes as long as 70 FP32 ones).
__device__ __forceinline__ double square_total(float2 hi, float2 mid, float2 lo) {
    float2 e;   // of (hi, mid)
    const float2 s = two_sum(make_float2(hi.x, mid.x), make_float2(hi.y, mid.y), e);
    return (double)s.x + (((double)s.y + (double)e.x) + (double)(e.y + (lo.x + lo.y)));
}

// One orientation per block: transform I0, and for every PSF c the energy B_c = sum_{k != 0} w_kx |F T_c|^2 (of
// the FP32 products that are stored) and the normalised product.
// GB300's float64 rate is 1/70 of its FP32 rate, and squaring every product in float64 (two conversions
// and three operations) took most of the kernel's 1.5 us per orientation (128 px, 8 PSFs). Each thread sums
// its squares in FP32 triples, exact beyond float64's own rounding, and the threads' sums are added in float64 by
// pairs: error of B 1.0e-16 (rms over models, PSFs and sizes), as with float64 throughout. (In FP32 pairs, restarted
// every 11 coefficients, 1e-15: the energy lies in few coefficients, so the runs' errors do not average.)
// The products are scaled by a power of two so that the largest |F| is near 1; a B so small against it that
// squares may have lost bits to underflow (below kSmall) is summed again in float64 throughout.
constexpr int kPsfChunk = 16;   // PSFs whose energies are reduced together
constexpr double kSmall = 1e-12;

template <int N>
__device__ __forceinline__ double psf_energy64(const float2* F, const float* __restrict__ T) {
    double e = 0.0;
    for (int o = threadIdx.x; o < N * Dft<N>::H; o += Dft<N>::T) e += half_energy<N>(o, c_scale(F[o], __ldg(T + o)));
    return e;
}

template <int N>
__global__ void __launch_bounds__(Dft<N>::T, N == 192 ? 1 : 2) k_psf_spectra(const float* __restrict__ img0,
                                                           const float2* __restrict__ g_tw,
                                                           const float* __restrict__ T, int nctf,
                                                           float2* __restrict__ spec,
                                                           double* __restrict__ kB, float* __restrict__ amax,
                                                           int* __restrict__ status) {
    constexpr int H = Dft<N>::H, TH = Dft<N>::T, PER = Dft<N>::PER;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double part[kPsfChunk][TH / 32];
    __shared__ float scale[kPsfChunk];   // 1 / sqrt(B); -1 where B is to be summed in float64
    const DftSm<N> sm(smem);
    const int q = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    sm.twiddles(g_tw, false);
    __syncthreads();
    r2c_rows<N>(img0 + (size_t)q * N * N, 0.f, sm);
    __syncthreads();
    c2c_columns_inplace<N>(sm);
    // power of two near 1 / max |F| over k != 0 (1 for an empty or non-finite spectrum)
    float fm = 0.f;
    for (int o = threadIdx.x; o < N * H; o += TH)
        if (o > 0) fm = fmaxf(fm, fmaxf(fabsf(sm.F[o].x), fabsf(sm.F[o].y)));
    fm = block_max<TH>(fm, reinterpret_cast<float*>(sm.red));
    int ex = 0;
    if (fm > 0.f && fm < INFINITY) frexpf(fm, &ex);
    ex = max(-120, min(120, ex));
    const float sc = ldexpf(1.f, -ex);
    for (int c0 = 0; c0 < nctf; c0 += kPsfChunk) {
        const int nc = min(kPsfChunk, nctf - c0);
        for (int c = 0; c < nc; ++c) {
            const float* Tc = T + (size_t)(c0 + c) * N * H;
            const float2 none = make_float2(0.f, 0.f);
            float2 hi = none, mid = none, lo = none;   // of the real and the imaginary parts
            // unrolled as a whole, so that the PSF's values are loaded ahead (in runs of 11, each waited for, the 128
            // orientations x 8 PSFs of a re-ranking wave took 172 us instead of 119)
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                const int o = threadIdx.x + i * TH;
                if (o < N * H) {
                    const int kx = o % H;
                    float2 v = c_scale(c_scale(sm.F[o], __ldg(Tc + o)), sc);
                    if (o == 0) v = make_float2(0.f, 0.f);   // DC (see half_energy)
                    const float w = kx == 0 || kx == N / 2 ? 1.f : 2.f;
                    add_square(hi, mid, lo, v, make_float2(w, w));
                }
            }
            double e = square_total(hi, mid, lo);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) e += __shfl_xor_sync(0xffffffffu, e, off);
            if (lane == 0) part[c][warp] = e;
        }
        __syncthreads();
        // the warps' sums, the scale and ln B of a PSF by one lane (float64 by every thread takes longer than the sums)
        if (threadIdx.x < nc) {
            const int c = threadIdx.x;
            double t[TH / 32];
#pragma unroll
            for (int w = 0; w < TH / 32; ++w) t[w] = part[c][w];
#pragma unroll
            for (int n = TH / 64; n > 0; n /= 2)
#pragma unroll
                for (int w = 0; w < n; ++w) t[w] = t[2 * w] + t[2 * w + 1];
            const bool sure = t[0] > kSmall && t[0] < INFINITY;
            const double B = ldexp(t[0], 2 * ex);
            scale[c] = sure ? (float)(1.0 / sqrt(B)) : -1.f;
            if (sure) kB[(size_t)q * nctf + c0 + c] = -0.5 * log(B);
        }
        __syncthreads();
        for (int c = 0; c < nc; ++c) {
            const float* Tc = T + (size_t)(c0 + c) * N * H;
            const size_t p = (size_t)q * nctf + c0 + c;
            float sB = scale[c];
            if (sB < 0.f) {   // uniform over the block
                double B = psf_energy64<N>(sm.F, Tc), dummy = 0.0;
                block_sum2<TH>(B, dummy, sm.red);
                const bool bad = !(B > 0.0);   // B = n C_cc - C_c^2 (Plancherel)
                sB = bad ? 0.f : (float)(1.0 / sqrt(B));
                if (threadIdx.x == 0) {
                    if (bad) atomicOr(status, BIOEM_DEV_NUMERIC);
                    kB[p] = bad ? -INFINITY : -0.5 * log(B);
                }
            }
            const float mx = block_max<TH>(store_half_spectrum<N>(sm.F, Tc, sB, spec + p * N * H),
                                           reinterpret_cast<float*>(sm.red));
            if (threadIdx.x == 0) amax[p] = mx;
        }
    }
}

// ---- transforms by factors, for the maps
// cos(2 pi j / n), by the Taylor series of cos or sin about 0 after reduction to an eighth of a turn.
constexpr double cos_turn(int j, int n) {
    double x = (double)(((j % n) + n) % n) / n;
    if (x > 0.5) x = 1.0 - x;
    double sign = 1.0;
    if (x > 0.25) {
        x = 0.5 - x;
        sign = -1.0;
    }
    const bool use_sin = x > 0.125;
    const double t = 2.0 * 3.14159265358979323846 * (use_sin ? 0.25 - x : x);
    double term = use_sin ? t : 1.0, sum = 0.0;
    for (int k = use_sin ? 2 : 1; k < 30; k += 2) {
        sum += term;
        term *= -t * t / (k * (k + 1));
    }
    return sign * sum;
}
// w.x, w.y[j] = cos, sin of 2 pi j / R
template <int R>
struct Roots {
    float c[R] = {}, s[R] = {};
    constexpr Roots() {
        for (int j = 0; j < R; ++j) {
            c[j] = (float)cos_turn(j, R);
            s[j] = (float)cos_turn(4 * j - R, 4 * R);
        }
    }
};
// v exp(-+ 2 pi i j / R) (upper sign forward), 0 <= j < R known at compile time
template <int R, bool INV>
__device__ __forceinline__ float2 turn(float2 v, int j) {
    constexpr Roots<R> w{};
    if (j == 0) return v;
    if (4 * j == R) return INV ? make_float2(-v.y, v.x) : make_float2(v.y, -v.x);
    if (2 * j == R) return make_float2(-v.x, -v.y);
    return INV ? c_mul(v, make_float2(w.c[j], w.s[j])) : c_mul(v, make_float2(w.c[j], -w.s[j]));
}
// In-register transform of R = 2^a or 3 2^a values, natural order in and out.
template <int R, bool INV>
__device__ __forceinline__ void dft(float2 (&x)[R]) {
    if constexpr (R == 2) {
        const float2 a = x[0];
        x[0] = c_add(a, x[1]);
        x[1] = c_sub(a, x[1]);
    } else if constexpr (R == 3) {
        const float2 t = c_add(x[1], x[2]), d = c_sub(x[1], x[2]);
        const float2 m = make_float2(fmaf(-0.5f, t.x, x[0].x), fmaf(-0.5f, t.y, x[0].y));
        constexpr float s = INV ? 0.8660254037844386f : -0.8660254037844386f;
        x[0] = c_add(x[0], t);
        x[1] = make_float2(fmaf(-s, d.y, m.x), fmaf(s, d.x, m.y));
        x[2] = make_float2(fmaf(s, d.y, m.x), fmaf(-s, d.x, m.y));
    } else if constexpr (R == 4) {
        const float2 a = c_add(x[0], x[2]), b = c_sub(x[0], x[2]), c = c_add(x[1], x[3]);
        const float2 d = turn<4, INV>(c_sub(x[1], x[3]), 1);
        x[0] = c_add(a, c);
        x[1] = c_add(b, d);
        x[2] = c_sub(a, c);
        x[3] = c_sub(b, d);
    } else {
        constexpr int P = R % 4 == 0 ? 4 : 2, Q = R / P;
        float2 y[Q][P];
#pragma unroll
        for (int b = 0; b < Q; ++b) {
#pragma unroll
            for (int a = 0; a < P; ++a) y[b][a] = x[Q * a + b];
            dft<P, INV>(y[b]);
#pragma unroll
            for (int k = 0; k < P; ++k) y[b][k] = turn<R, INV>(y[b][k], b * k);
        }
#pragma unroll
        for (int k = 0; k < P; ++k) {
            float2 t[Q];
#pragma unroll
            for (int b = 0; b < Q; ++b) t[b] = y[b][k];
            dft<Q, INV>(t);
#pragma unroll
            for (int k2 = 0; k2 < Q; ++k2) x[k + P * k2] = t[k2];
        }
    }
}

// N = 16 R: with n = R a + b and k = k1 + 16 k2, a length-N transform is R transforms of 16 values (over a),
// a turn by b k1 / N and 16 transforms of R values (over b).
template <int N>
struct Fft {
    static constexpr int R = N / 16, H = N / 2 + 1;
    static constexpr int T = N == 32 ? 64 : N == 64 ? 128 : N == 192 ? 512 : 256;
    static constexpr int MINB = N <= 64 ? 8 : N == 192 ? 1 : 3;
    // Rows 2p and 2p + 1 of the spectrum hold the packed transform of a pair of image rows meanwhile, R runs
    // of 16 with one place between them; with this pitch neither the runs nor the pairs conflict.
    static constexpr int P = 17 * R / 2;
    static_assert(R % 2 == 0 && P >= H, "a packed transform fits two rows");
    static constexpr size_t SMEM = (size_t)(N * P + N) * sizeof(float2);
};

// Synthetic map for pair i: I1 = Re F^-1[F(I0_i) T_i] with F^-1 normalised by 1/N^2.  A block per map, every pass in
// place in shared memory: rows two by two as one complex transform (a warp takes four pairs and needs no
// block barrier), columns with the PSF and the first half of the inverse applied while a column's R
// frequencies are in registers.  Bound by shared memory and the latency of its passes.  1024 maps at 128 px: 2174 us by
// dense sums over shared memory, 721 us by dense sums in register tiles (N multiply-adds per
// coefficient and pass), 65 us so.  The spectra that are scored keep the dense sums (k_psf_spectra): another
// rounding moves their FP32 scale.
template <int N>
__global__ void __launch_bounds__(Fft<N>::T, Fft<N>::MINB) k_psf_real(const float* __restrict__ img0,
                                                                   const float2* __restrict__ g_tw,
                                                                   const float* __restrict__ T,
                                                                   float* __restrict__ out) {
    using C = Fft<N>;
    constexpr int R = C::R, H = C::H, P = C::P, TH = C::T, NW = TH / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    float2* const F = reinterpret_cast<float2*>(smem);
    float2* const tw = F + N * P;   // exp(-2 pi i t / N)
    const size_t map = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < N; i += TH) tw[i] = g_tw[i];
    __syncthreads();
    // rows: C = row 2p + i row 2p + 1 transformed, then taken apart into the halves F (halved before the sums,
    // which would double the largest sum of an image that is within the FP32 range)
    const float* img = img0 + map * N * N;
    const int j = lane & 7, kA = j, kB = j ? 16 - j : 8;   // a lane's two residues k1, partners under k -> N - k
    for (int g = warp; g < N / 8; g += NW) {
        for (int t = lane; t < 4 * R; t += 32) {
            const int p = 4 * g + t / R, b = t % R;
            const float* row = img + (size_t)2 * p * N + b;
            float2 x[16];
#pragma unroll
            for (int a = 0; a < 16; ++a) x[a] = make_float2(__ldg(row + R * a), __ldg(row + N + R * a));
            dft<16, false>(x);
            float2* buf = F + (size_t)2 * p * P + 17 * b;
#pragma unroll
            for (int k = 0; k < 16; ++k) buf[k] = k ? c_mul(x[k], tw[b * k]) : x[k];
        }
        __syncwarp();
        float2* const buf = F + (size_t)2 * (4 * g + (lane >> 3)) * P;
        float2 u[R], v[R];
#pragma unroll
        for (int b = 0; b < R; ++b) {
            u[b] = buf[17 * b + kA];
            v[b] = buf[17 * b + kB];
        }
        dft<R, false>(u);
        dft<R, false>(v);
        __syncwarp();
        auto apart = [&](int k, float2 c, float2 d) {   // d = C(N - k)
            buf[k] = make_float2(fmaf(0.5f, c.x, 0.5f * d.x), fmaf(0.5f, c.y, -0.5f * d.y));
            buf[P + k] = make_float2(fmaf(0.5f, c.y, 0.5f * d.y), fmaf(0.5f, d.x, -0.5f * c.x));
        };
#pragma unroll
        for (int k2 = 0; k2 < R / 2; ++k2) {
            apart(kA + 16 * k2, u[k2], j ? v[R - 1 - k2] : u[(R - k2) % R]);
            apart(kB + 16 * k2, v[k2], j ? u[R - 1 - k2] : v[R - 1 - k2]);
        }
        if (j == 0) apart(N / 2, u[R / 2], u[R / 2]);
    }
    __syncthreads();
    // columns
    for (int e = threadIdx.x; e < H * R; e += TH) {
        const int kx = e % H, b = e / H;
        float2* col = F + b * P + kx;
        float2 x[16];
#pragma unroll
        for (int a = 0; a < 16; ++a) x[a] = col[R * a * P];
        dft<16, false>(x);
#pragma unroll
        for (int k = 0; k < 16; ++k) col[R * k * P] = k ? c_mul(x[k], tw[b * k]) : x[k];
    }
    __syncthreads();
    const float* Ti = T + map * N * H;
    for (int e = threadIdx.x; e < H * 16; e += TH) {
        const int kx = e % H, k1 = e / H;
        float2* col = F + R * k1 * P + kx;
        float2 v[R];
#pragma unroll
        for (int b = 0; b < R; ++b) v[b] = col[b * P];
        dft<R, false>(v);
#pragma unroll
        for (int k2 = 0; k2 < R; ++k2) v[k2] = c_scale(v[k2], __ldg(Ti + (k1 + 16 * k2) * H + kx));
        dft<R, true>(v);
#pragma unroll
        for (int b = 0; b < R; ++b) col[b * P] = b ? c_mulc(tw[b * k1], v[b]) : v[b];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < H * R; e += TH) {
        const int kx = e % H, b = e / H;
        float2* col = F + b * P + kx;
        float2 x[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] = col[R * k * P];
        dft<16, true>(x);
#pragma unroll
        for (int a = 0; a < 16; ++a) col[R * a * P] = x[a];
    }
    __syncthreads();
    // rows: C(k) = G_2p(k) + i G_2p+1(k) of the Hermitian rows G (the imaginary parts at k = 0 and N/2 do not
    // count), transformed back: its real and imaginary parts are the two rows of the map
    constexpr float inv = 1.f / ((float)N * N);
    float* o = out + map * N * N;
    for (int g = warp; g < N / 8; g += NW) {
        float2* const buf = F + (size_t)2 * (4 * g + (lane >> 3)) * P;
        float2 u[R], v[R], dA[R / 2], dB[R / 2];
        auto join = [&](int k, float2& c, float2& d) {
            const float2 g0 = buf[k], g1 = buf[P + k];
            c = make_float2(g0.x - g1.y, g0.y + g1.x);
            d = make_float2(g0.x + g1.y, g1.x - g0.y);   // C(N - k)
        };
#pragma unroll
        for (int k2 = 0; k2 < R / 2; ++k2) {
            join(kA + 16 * k2, u[k2], dA[k2]);
            join(kB + 16 * k2, v[k2], dB[k2]);
        }
        const float2 mid = make_float2(buf[N / 2].x, buf[P + N / 2].x);
        if (j == 0) u[0] = make_float2(buf[0].x, buf[P].x);
#pragma unroll
        for (int i = R / 2; i < R; ++i) {
            u[i] = j ? dB[R - 1 - i] : i == R / 2 ? mid : dA[(R - i) % (R / 2)];
            v[i] = j ? dA[R - 1 - i] : dB[R - 1 - i];
        }
        dft<R, true>(u);
        dft<R, true>(v);
        __syncwarp();
#pragma unroll
        for (int b = 0; b < R; ++b) {
            buf[17 * b + kA] = c_mulc(tw[b * kA], u[b]);
            buf[17 * b + kB] = c_mulc(tw[b * kB], v[b]);
        }
        __syncwarp();
        for (int t = lane; t < 4 * R; t += 32) {
            const int p = 4 * g + t / R, b = t % R;
            const float2* run = F + (size_t)2 * p * P + 17 * b;
            float2 x[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) x[k] = run[k];
            dft<16, true>(x);
            float* row = o + (size_t)2 * p * N + b;
#pragma unroll
            for (int a = 0; a < 16; ++a) {
                row[R * a] = x[a].x * inv;
                row[N + R * a] = x[a].y * inv;
            }
        }
        __syncwarp();
    }
}

// Real-space image of a stored unit-norm half spectrum S (Eq. 3, inverse transform):
//   x(r) = Re sum_k w_kx S(k) exp(+2 pi i k.r / N),  w = 1 on kx = 0, N/2 and 2 elsewhere,
// rescaled to unit norm (float64 sum of squares); zero-mean because S(0) = 0.  With the forward
// transforms above this is the zero-mean, unit-norm image whose correlations the scoring kernels
// evaluate: sum_r o'(r) c'(r + d) = rho(d).  Writes x [N][N] and max |x|.
template <int N>
__global__ void __launch_bounds__(Dft<N>::T) k_spec_to_real(const float2* __restrict__ spec,
                                                           const float2* __restrict__ g_tw, float* __restrict__ out,
                                                           float* __restrict__ amax) {
    constexpr int H = Dft<N>::H, TH = Dft<N>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    const DftSm<N> sm(smem);
    const int i = blockIdx.x;
    sm.twiddles(g_tw, true);
    const float2* S = spec + (size_t)i * N * H;
    for (int o = threadIdx.x; o < N * H; o += TH) sm.F[o] = S[o];
    __syncthreads();
    c2c_columns_inplace<N>(sm);
    sm.twiddles(g_tw, false);
    __syncthreads();
    float* xo = out + (size_t)i * N * N;
    double e = 0.0, dummy = 0.0;
    c2r_rows<N>(sm, [&](int y, int x, float v) {
        xo[y * N + x] = v;
        e += (double)v * v;
    });
    block_sum2<TH>(e, dummy, sm.red);   // its barriers also order the stores before the reads below
    const float scale = e > 0.0 ? (float)(1.0 / sqrt(e)) : 0.f;
    float mx = 0.f;
    for (int p = threadIdx.x; p < N * N; p += TH) {
        const float r = xo[p] * scale;
        xo[p] = r;
        mx = fmaxf(mx, fabsf(r));
    }
    mx = block_max<TH>(mx, reinterpret_cast<float*>(sm.red));
    if (threadIdx.x == 0) amax[i] = mx;
}

// Sets the dynamic shared memory limit where it is needed: a block may use 48 KB, static variables (up to 4 KB in
// these kernels) included, without it, and the call takes 1 us of a small image's 15.
template <int N>
int set_smem(const void* fn, size_t bytes) {
    if (bytes <= 40 * 1024) return 0;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess ? 0 : -1;
}

void ctf_coefficients(const bioem_ctf& c, double* out4) {
    const double v = c.voltage_kV * 1.0e3;
    const double lam = 12.2643 / sqrt(v * (1.0 + 0.97845e-6 * v));
    out4[0] = lam * c.defocus_A / (2.0 * 3.14159265358979323846);
    out4[1] = c.amp_contrast;
    out4[2] = c.bfactor_A2 / (8.0 * 3.14159265358979323846 * 3.14159265358979323846);
    out4[3] = sqrt(1.0 - c.amp_contrast * c.amp_contrast);
}

// Build the CTF table for nctf PSFs into *d_T (allocated here; caller frees).
int build_ctf_table(bioem_ctx* ctx, const bioem_ctf* ctfs, int nctf, int npix, double pixel_A, float** d_T) {
    double* h = (double*)malloc(sizeof(double) * 4 * nctf);
    if (!h) return bioem_set_error(ctx, BIOEM_ERR_OOM, "host allocation failed");
    for (int c = 0; c < nctf; ++c) ctf_coefficients(ctfs[c], h + 4 * c);
    double* d_coef = nullptr;
    cudaError_t e = cudaMallocAsync((void**)&d_coef, sizeof(double) * 4 * nctf, ctx->stream);
    if (e != cudaSuccess) { free(h); return bioem_set_error(ctx, BIOEM_ERR_OOM, "cudaMallocAsync(ctf coef)"); }
    const size_t tsize = (size_t)nctf * npix * (npix / 2 + 1);
    e = cudaMallocAsync((void**)d_T, sizeof(float) * tsize, ctx->stream);
    if (e != cudaSuccess) {
        cudaFreeAsync(d_coef, ctx->stream);
        free(h);
        return bioem_set_error(ctx, BIOEM_ERR_OOM, "cudaMallocAsync(ctf table)");
    }
    e = cudaMemcpyAsync(d_coef, h, sizeof(double) * 4 * nctf, cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) {
        const size_t work = (tsize / 4 + 255) / 256 + 1;
        const int blocks = (int)(work < 4096 ? work : 4096);
        bioem_launch_begin(ctx, KID_CTF_TABLE);
        k_ctf_table<<<blocks, 256, 0, ctx->stream>>>(d_coef, nctf, npix, pixel_A, *d_T);
        e = cudaGetLastError();
        bioem_launch_end(ctx, KID_CTF_TABLE);
    }
    // the copy reads h asynchronously from pageable memory: it has completed once the call returns
    cudaFreeAsync(d_coef, ctx->stream);
    free(h);
    if (e != cudaSuccess) {
        cudaFreeAsync(*d_T, ctx->stream);
        *d_T = nullptr;
        return bioem_check_cuda(ctx, e, "ctf table");
    }
    return BIOEM_OK;
}

template <int N>
int launch_prepare_n(bioem_ctx* ctx, const float* d_images, bioem_images* im) {
    const size_t sm = DftSm<N>::bytes();
    auto kern = (uintptr_t)d_images % 16 == 0 ? k_prepare_images<N, true> : k_prepare_images<N, false>;
    if (set_smem<N>((const void*)kern, sm)) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "smem attribute");
    const double cn = bioem_log_norm_constant(N * N);
    bioem_launch_begin(ctx, KID_PREPARE);
    kern<<<im->n_img, Dft<N>::T, sm, ctx->stream>>>(d_images, bioem_twiddles(ctx, N), im->d_spec, im->d_kA,
                                                    im->d_amax, cn, ctx->d_status);
    bioem_launch_end(ctx, KID_PREPARE);
    return bioem_check_cuda(ctx, cudaGetLastError(), "k_prepare_images");
}

template <int N>
int launch_project_n(bioem_ctx* ctx, const float* d_atoms, int n_atoms, double sigma_A, const float* d_quats,
                     int nq, const bioem_ctf* ctfs, int nctf, bioem_projset* ps) {
    float* d_T = nullptr;
    int rc = build_ctf_table(ctx, ctfs, nctf, N, ps->pixel_A, &d_T);
    if (rc) return rc;
    // orientations in waves bounded to ~1 GiB of I0 scratch
    const int wave = (int)((1ull << 30) / ((size_t)N * N * sizeof(float)));
    const int qw = nq < wave ? nq : wave;
    float* d_I0 = nullptr;
    if (cudaMallocAsync((void**)&d_I0, sizeof(float) * (size_t)qw * N * N, ctx->stream) != cudaSuccess) {
        cudaFreeAsync(d_T, ctx->stream);
        return bioem_set_error(ctx, BIOEM_ERR_OOM, "cudaMallocAsync(projection scratch)");
    }
    const size_t sm = DftSm<N>::bytes();
    if (set_smem<N>((const void*)k_project<N>, ProjCfg<N>::SMEM) || set_smem<N>((const void*)k_psf_spectra<N>, sm)) rc = bioem_set_error(ctx, BIOEM_ERR_CUDA, "smem attribute");
    for (int q0 = 0; q0 < nq && rc == BIOEM_OK; q0 += qw) {
        const int nb = nq - q0 < qw ? nq - q0 : qw;
        bioem_launch_begin(ctx, KID_PROJECT);
        k_project<N><<<nb, ProjCfg<N>::T, ProjCfg<N>::SMEM, ctx->stream>>>(reinterpret_cast<const float4*>(d_atoms), n_atoms,
                                                        reinterpret_cast<const float4*>(d_quats) + q0, sigma_A,
                                                        ps->pixel_A, window_reach(sigma_A, ps->pixel_A), d_I0);
        bioem_launch_end(ctx, KID_PROJECT);
        rc = bioem_check_cuda(ctx, cudaGetLastError(), "k_project");
        if (rc) break;
        const size_t p0 = (size_t)q0 * nctf;
        bioem_launch_begin(ctx, KID_PSF_SPECTRA);
        k_psf_spectra<N><<<nb, Dft<N>::T, sm, ctx->stream>>>(d_I0, bioem_twiddles(ctx, N), d_T, nctf,
                                                             ps->d_spec + p0 * N * (N / 2 + 1), ps->d_kB + p0,
                                                             ps->d_amax + p0, ctx->d_status);
        bioem_launch_end(ctx, KID_PSF_SPECTRA);
        rc = bioem_check_cuda(ctx, cudaGetLastError(), "k_psf_spectra");
    }
    cudaFreeAsync(d_I0, ctx->stream);
    cudaFreeAsync(d_T, ctx->stream);
    return rc;
}

template <int N>
int launch_synthetic_n(bioem_ctx* ctx, const float* d_atoms, int n_atoms, double sigma_A, const float* d_quats,
                       const bioem_ctf* ctfs, int n, double pixel_A, float* d_out) {
    float* d_T = nullptr;
    int rc = build_ctf_table(ctx, ctfs, n, N, pixel_A, &d_T);
    if (rc) return rc;
    float* d_I0 = nullptr;
    if (cudaMallocAsync((void**)&d_I0, sizeof(float) * (size_t)n * N * N, ctx->stream) != cudaSuccess) {
        cudaFreeAsync(d_T, ctx->stream);
        return bioem_set_error(ctx, BIOEM_ERR_OOM, "cudaMallocAsync(synthetic scratch)");
    }
    if (set_smem<N>((const void*)k_project<N>, ProjCfg<N>::SMEM)) {
        cudaFreeAsync(d_I0, ctx->stream);
        cudaFreeAsync(d_T, ctx->stream);
        return bioem_set_error(ctx, BIOEM_ERR_CUDA, "smem attribute");
    }
    bioem_launch_begin(ctx, KID_PROJECT);
    k_project<N><<<n, ProjCfg<N>::T, ProjCfg<N>::SMEM, ctx->stream>>>(reinterpret_cast<const float4*>(d_atoms), n_atoms,
                                                   reinterpret_cast<const float4*>(d_quats), sigma_A, pixel_A,
                                                   window_reach(sigma_A, pixel_A), d_I0);
    bioem_launch_end(ctx, KID_PROJECT);
    rc = bioem_check_cuda(ctx, cudaGetLastError(), "k_project");
    if (!rc && set_smem<N>((const void*)k_psf_real<N>, Fft<N>::SMEM)) rc = bioem_set_error(ctx, BIOEM_ERR_CUDA, "smem attribute");
    if (!rc) {
        bioem_launch_begin(ctx, KID_PSF_REAL);
        k_psf_real<N><<<n, Fft<N>::T, Fft<N>::SMEM, ctx->stream>>>(d_I0, bioem_twiddles(ctx, N), d_T, d_out);
        bioem_launch_end(ctx, KID_PSF_REAL);
        rc = bioem_check_cuda(ctx, cudaGetLastError(), "k_psf_real");
    }
    cudaFreeAsync(d_I0, ctx->stream);
    cudaFreeAsync(d_T, ctx->stream);
    return rc;
}

template <int N>
int launch_spec_to_real_n(bioem_ctx* ctx, const float2* spec, int count, float* out, float* amax) {
    const size_t sm = DftSm<N>::bytes();
    if (set_smem<N>((const void*)k_spec_to_real<N>, sm)) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "smem attribute");
    bioem_launch_begin(ctx, KID_GEMM_OPS);
    k_spec_to_real<N><<<count, Dft<N>::T, sm, ctx->stream>>>(spec, bioem_twiddles(ctx, N), out, amax);
    bioem_launch_end(ctx, KID_GEMM_OPS);
    return bioem_check_cuda(ctx, cudaGetLastError(), "k_spec_to_real");
}

}  // namespace

double bioem_log_norm_constant(int n) {
    const double nn = n;
    return -log(2.0) + (1.0 - nn / 2.0) * log(2.0 * 3.14159265358979323846) + lgamma((nn - 3.0) / 2.0) +
           (nn - 3.0) / 2.0 * log(2.0 * nn);
}

#define BIOEM_DISPATCH_N(npix, CALL)                                          \
    switch (npix) {                                                           \
        case 32: return CALL(32);                                             \
        case 64: return CALL(64);                                             \
        case 96: return CALL(96);                                             \
        case 128: return CALL(128);                                           \
        case 192: return CALL(192);                                           \
        default: return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE, "unsupported image size %d", npix); \
    }

int bioem_launch_prepare(bioem_ctx* ctx, const float* d_images, bioem_images* im) {
#define CALL(N) launch_prepare_n<N>(ctx, d_images, im)
    BIOEM_DISPATCH_N(im->nx, CALL)
#undef CALL
}

int bioem_launch_project(bioem_ctx* ctx, const float* d_atoms, int n_atoms, double sigma_A, const float* d_quats,
                         int nq, const bioem_ctf* ctfs, int nctf, bioem_projset* ps) {
#define CALL(N) launch_project_n<N>(ctx, d_atoms, n_atoms, sigma_A, d_quats, nq, ctfs, nctf, ps)
    BIOEM_DISPATCH_N(ps->nx, CALL)
#undef CALL
}

int bioem_launch_spec_to_real(bioem_ctx* ctx, const float2* spec, int count, int npix, float* out, float* amax) {
    if (count <= 0) return BIOEM_OK;
#define CALL(N) launch_spec_to_real_n<N>(ctx, spec, count, out, amax)
    BIOEM_DISPATCH_N(npix, CALL)
#undef CALL
}

int bioem_launch_synthetic(bioem_ctx* ctx, const float* d_atoms, int n_atoms, double sigma_A, const float* d_quats,
                           const bioem_ctf* ctfs, int n, int npix, double pixel_A, float* d_out) {
#define CALL(N) launch_synthetic_n<N>(ctx, d_atoms, n_atoms, sigma_A, d_quats, ctfs, n, pixel_A, d_out)
    BIOEM_DISPATCH_N(npix, CALL)
#undef CALL
}

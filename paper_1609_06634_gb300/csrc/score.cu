// Fused scoring kernel: per (image, parameter set) pair, the Fourier-space product, the inverse
// transform evaluated on the displacement window only, and the closed-form likelihood with a
// log-sum-exp over displacements (Sec. 3.3, Eqs. 11-12; Sec. 3.9 and Sec. 5 note that the product,
// the inverse FFT and the likelihood were three kernels with the correlation map stored between
// them, and that only some output coefficients are needed: here they are one kernel and the map
// never leaves the SM).
//
// Spectra (both unit-norm, DC = 0, half spectrum kx = 0..N/2):
//   rho(d) = X(d) / sqrt(A B) = Re sum_{ky} sum_{kx<=N/2} w_kx conj(O(k)) C(k) exp(+2 pi i k.d / N)
// with w = 1 on the kx = 0 and kx = N/2 columns, 2 elsewhere.  Evaluated in two stages:
//   stage A (per column kx, along ky):  Q(dy, kx) = sum_ky conj(O) C exp(+2 pi i ky dy / N)
//   stage B (per row dy, along kx):     rho(dy, dx) = Re sum_kx w_kx Q(dy, kx) exp(+2 pi i kx dx / N)
// each as a pruned transform: the N (or N/2) inputs split into R interleaved sub-sequences of
// length L = 16, each transformed by an in-register radix-2 FFT, then recombined with twiddles for
// the 2 SMAX + 1 wanted outputs only.
//
// Likelihood (closed form of Eq. 8 integrated over N, mu, lambda):
//   ln L(d) = kA + kB + (3 - n)/2 ln(1 - rho(d)^2),  kA = (3-n)/2 ln A + c(n),  kB = -1/2 ln B.
// Per pair the kernel records t_min = min_d ln(1 - rho^2), s = sum_d exp((3-n)/2 (t(d) - t_min))
// and the argmin d; a float64 reduction (k_reduce_wave) turns the records into per-image and
// per-orientation log-sum-exps and maximising parameters.
#include <math.h>
#include <stdio.h>

#include <mutex>
#include <type_traits>

#include "bioem_internal.cuh"
#include "rdft16.cuh"

namespace {

constexpr int L = 16;   // sub-transform length
// Dynamic shared memory a scoring block may take: 227 KiB per block, less 1 KiB for the kernels'
// static shared variables.
constexpr size_t kScoreSmemLimit = 227u * 1024u - 1024u;

// W_M^t = exp(+2 pi i t / M), uploaded once per device.
__constant__ float2 c_w16[16];
__constant__ float2 c_w32[32];
__constant__ float2 c_w64[64];
__constant__ float2 c_w128[128];
__constant__ float2 c_w96[96];
__constant__ float2 c_w192[192];

template <int M>
__device__ __forceinline__ float2 cw(int t) {
    if constexpr (M == 16) return c_w16[t];
    else if constexpr (M == 32) return c_w32[t];
    else if constexpr (M == 64) return c_w64[t];
    else if constexpr (M == 96) return c_w96[t];
    else if constexpr (M == 192) return c_w192[t];
    else return c_w128[t];
}

template <int M>
__device__ __forceinline__ const float2* cw_table() {
    if constexpr (M == 16) return c_w16;
    else if constexpr (M == 32) return c_w32;
    else if constexpr (M == 64) return c_w64;
    else if constexpr (M == 96) return c_w96;
    else if constexpr (M == 192) return c_w192;
    else return c_w128;
}

// d * W_LL^t for a compile-time exponent t < LL / 2.
template <int LL, int T>
__device__ __forceinline__ float2 twiddle_mul(float2 d) {
    if constexpr (T == 0) {
        return d;
    } else if constexpr (4 * T == LL) {          // W^(LL/4) = i
        return make_float2(-d.y, d.x);
    } else if constexpr (8 * T == LL) {          // (1 + i) / sqrt 2
        const float r = 0.70710678118654752f;
        return make_float2((d.x - d.y) * r, (d.x + d.y) * r);
    } else if constexpr (8 * T == 3 * LL) {      // (-1 + i) / sqrt 2
        const float r = 0.70710678118654752f;
        return make_float2(-(d.x + d.y) * r, (d.x - d.y) * r);
    } else {
        return c_mul(d, cw<LL>(T));
    }
}

template <int LL, int HALF, int BLK, int J>
__device__ __forceinline__ void dif_butterflies(float2 (&x)[LL]) {
    if constexpr (BLK < LL) {
        if constexpr (J < HALF) {
            const float2 a = x[BLK + J], b = x[BLK + J + HALF];
            x[BLK + J] = __fadd2_rn(a, b);
            x[BLK + J + HALF] = twiddle_mul<LL, J * (LL / (2 * HALF))>(__ffma2_rn(b, make_float2(-1.f, -1.f), a));
            dif_butterflies<LL, HALF, BLK, J + 1>(x);
        } else {
            dif_butterflies<LL, HALF, BLK + 2 * HALF, 0>(x);
        }
    }
}

template <int LL, int HALF>
__device__ __forceinline__ void dif_stages(float2 (&x)[LL]) {
    if constexpr (HALF >= 1) {
        dif_butterflies<LL, HALF, 0, 0>(x);
        dif_stages<LL, HALF / 2>(x);
    }
}

// In-register DFT y[u] = sum_a x[a] W_LL^(a u), radix-2 decimation in frequency; on return
// y[u] is stored at x[bitrev(u)].
template <int LL>
__device__ __forceinline__ void fft_dif(float2 (&x)[LL]) {
    dif_stages<LL, LL / 2>(x);
}

template <int LL, int J>
__device__ __forceinline__ void first_stage_half_zero(float2 (&x)[LL]) {
    if constexpr (J < LL / 2) {
        x[J + LL / 2] = twiddle_mul<LL, J>(x[J]);
        first_stage_half_zero<LL, J + 1>(x);
    }
}

// fft_dif for inputs whose upper half x[LL/2 ..] is zero: the first stage's butterflies reduce to
// copies (a + 0 = a, a - 0 = a).
template <int LL>
__device__ __forceinline__ void fft_dif_half_zero(float2 (&x)[LL]) {
    first_stage_half_zero<LL, 0>(x);
    dif_stages<LL, LL / 4>(x);
}

__host__ __device__ constexpr int bitrev(int u, int bits) {
    int r = 0;
    for (int i = 0; i < bits; ++i) r |= ((u >> i) & 1) << (bits - 1 - i);
    return r;
}
__host__ __device__ constexpr int ilog2(int v) { return v <= 1 ? 0 : 1 + ilog2(v / 2); }
__host__ __device__ constexpr int pmod(int a, int m) { return ((a % m) + m) % m; }

template <int N_, int SMAX_, int NG_, int GT_, int GPB_, bool PACK_, int BSPLIT_ = 1, int ASPLIT_ = 1>
struct Cfg {
    static constexpr int N = N_;
    static constexpr int SMAX = SMAX_;
    static constexpr int NC = N / 2;
    static constexpr int H = NC + 1;           // half-spectrum row length (kx = 0..N/2)
    static constexpr int NS = 2 * SMAX + 1;    // displacements per axis
    static constexpr int NROW = 2 * SMAX;      // stage-B transform rows per pair (dy < SMAX)
    static constexpr int R = N / L;            // sub-sequences per transform
    static_assert(N % L == 0, "sub-transform length divides N");
    // Decoupled groups: the block's threads form NGROUP groups of GT threads.  A group takes batches of
    // GPB pairs from the item's counter and runs all their phases (packed edge columns, stage A, stage B,
    // the dy = +SMAX row, the combine) by itself, waiting only on its own named barrier, so that one
    // group's projection loads, barrier waits and short phases overlap the others' transform arithmetic.
    // The image spectrum and the twiddle tables are shared by the block.
    static constexpr int NGROUP = NG_, GT = GT_, GPB = GPB_;
    static constexpr int THREADS = NGROUP * GT;
    static constexpr int PB = NGROUP * GPB;    // pairs in flight per block
    static_assert(GT % 32 == 0 && THREADS <= 1024 && NGROUP <= 15, "whole warps; named barriers 1 .. 15");
    // stage-B threads per row: 2 when the group has two threads for every row (each sums half of the
    // sub-sequences, the halves are exchanged by a lane shuffle, and each evaluates the likelihood
    // for half of the dx outputs)
    static constexpr int BSPLIT = BSPLIT_;
    static constexpr int ROWS = GPB * NROW * BSPLIT;   // stage-B tasks per batch
    static_assert(BSPLIT == 1 || (BSPLIT == 2 && ROWS <= GT && ROWS % 32 == 0), "split rows: one per thread, whole warps");
    // stage-A threads per column: with 2 each sums half of the sub-sequences and they add their halves in
    // shared memory (twice the warps where shared memory holds few pairs; another order of the sums)
    static constexpr int ASPLIT = ASPLIT_;
    static_assert(ASPLIT == 1 || (ASPLIT == 2 && PACK_ && GPB * NC * 2 == GT && R % 2 == 0), "split columns: one per thread");
    static constexpr bool PREFETCH = THREADS <= 320;   // stage-A projection prefetch (registers)
    static constexpr int QS = H;               // Q row stride (complex); odd -> conflict-free columns
    static constexpr int NDIR = GPB * NS;      // outputs of the dy = +SMAX row, evaluated directly
    static constexpr size_t SM_IMG = (size_t)N * H * sizeof(float2);
    static constexpr size_t SM_Q = (size_t)PB * NS * QS * sizeof(float2);
    static constexpr size_t SM_QA = (SM_Q + 15) / 16 * 16;   // the twiddle table starts 16-byte aligned
    // twiddle table twc[b][d] = W_N^(b d), d = 0..SMAX (the outputs -d use the conjugate), rows of
    // an even length TWS so that pairs (d, d + 1), d even, are read as one 16-byte load
    static constexpr int TWS = 2 * ((SMAX + 2) / 2);
    // Packed edge columns: for real images and projections the product conj(O) C is Hermitian in
    // ky on the kx = 0 and kx = N/2 columns, so both columns' stage-A outputs are real, and one
    // complex transform of Z(ky) = P(ky, 0) + i P(ky, N/2) gives Q(dy, 0) as its real part and
    // Q(dy, N/2) as its imaginary part.  That leaves N/2 column tasks per pair; Z is formed for the
    // batch in shared memory before stage A.
    static constexpr bool PACK = PACK_;
    static constexpr int NCOL = PACK ? NC : H;      // stage-A column tasks per pair
    static constexpr int TASKS_A = GPB * NCOL;      // stage-A column tasks per batch (of ASPLIT threads)
    // with split columns Z shares its space with the stage-B pieces (a barrier more per batch)
    static constexpr bool ZALIAS = ASPLIT == 2;
    static constexpr size_t SM_ZB = PACK ? (size_t)PB * N * sizeof(float2) : 0;
    static constexpr size_t SM_Z = ZALIAS ? 0 : SM_ZB;
    // The dy = +SMAX row by real transforms (the 128 px, +-16 px instance): jobs (pair, Re / Im,
    // kx sub-sequence) on the last GPB 2 R threads of the group, each a real 16-point transform
    // recombined into the SMAX + 1 even (cosine) or odd (sine) outputs, summed over sub-sequences by
    // lane shuffles; a direct sum costs ~60 multiply-adds per output instead.
    static constexpr bool DIRFFT = PACK && N == 128 && SMAX == 16;
    static_assert(!DIRFFT || (GPB * NCOL == GT && BSPLIT == 2 && ((GPB * 2 * R) % 32 == 0 || GPB * 2 * R == 16)),
                  "each group's tasks on its own threads, its dy = +SMAX jobs on whole warps or half a warp");
    // The next batch's edge columns are formed while the rows of this one are transformed, by the threads without
    // a dy = +SMAX job (DIRFFT) or without a row or direct output.  As a step of their own before stage A, with a
    // barrier more, 128 px took 12.09 instead of 11.84 ns per pair at s = 16 and 6.87 instead of 6.55 at s = 4; by
    // all threads 11.92 and 6.72.
    static constexpr int ZFIRST = DIRFFT ? 0 : (ROWS + NDIR + 31) / 32 * 32 < GT ? (ROWS + NDIR + 31) / 32 * 32 : 0;
    static constexpr int ZCOUNT = DIRFFT ? GT - (GPB * 2 * R + 31) / 32 * 32 : GT - ZFIRST;
    // that instance keeps a second table 2 W_N^(b d) for stage B (the weight 2 of kx != 0 rides on the
    // twiddles, exact, instead of scaling every input)
    static constexpr bool TW2 = DIRFFT;
    static constexpr size_t SM_TWC = (size_t)(TW2 ? 2 : 1) * R * TWS * sizeof(float2);
    static_assert((SM_IMG + SM_QA) % 16 == 0 && (TWS * sizeof(float2)) % 16 == 0, "16-byte twiddle pairs");
    static constexpr size_t SM_ROW = (size_t)NGROUP * ROWS * (2 * sizeof(float) + sizeof(int));
    static constexpr size_t SM_DIR = (size_t)NGROUP * NDIR * sizeof(float);
    static constexpr size_t SM_TAIL = ZALIAS && SM_ZB > SM_ROW + SM_DIR ? SM_ZB : SM_ROW + SM_DIR;
    static constexpr size_t SM_BASE = (SM_IMG + SM_QA + SM_TWC + SM_Z + SM_TAIL + 7) / 8 * 8;
    static constexpr size_t SM_DTW = DIRFFT ? (size_t)2 * R * (SMAX + 1) * sizeof(float2) : 0;
    static constexpr size_t SM_DSUM = DIRFFT ? (size_t)PB * 2 * (SMAX + 1) * sizeof(float) : 0;
    // that row's twiddles in shared memory: ns per pair with them read through the L1 -> so: 64 px, s = 4: 2.20 ->
    // 2.15; 96 px 7.42 -> 7.19 (192 px 53 -> 62, whose strides share banks and whose L1 has fewer readers)
    static constexpr bool GTW = !DIRFFT && N < 192;
    static constexpr size_t SM_GTW = GTW ? (size_t)N * sizeof(float2) : 0;
    static constexpr size_t SMEM = SM_BASE + SM_DTW + SM_DSUM + SM_GTW;
    static_assert(SMEM <= kScoreSmemLimit, "dynamic shared memory per block");
    // Work by phases (k_score_phases) or by chunks from a counter (k_score).  Phases have fewer waits and end
    // evenly, but spread the blocks over all of a phase's spectra, which the instances with two pairs per group
    // feel: they read the most per second with the fewest warps.  ns per pair, chunks -> phases: 32 px 0.85 ->
    // 0.78; 64 px, s = 4: 2.16 -> 2.07, s = 8: 3.05 -> 2.90; 96 px 6.94 -> 6.85; 128 px, s = 4: 7.3 -> 6.87; but 128 px,
    // s = 16: 12.1 -> 12.4 (512 images: 11.59 -> 12.0); 192 px 49.2 -> 49.6 to 50.3.
    static constexpr bool PHASES = GPB > 2;
    // lanes that combine a pair's pieces (NROW BSPLIT rows and NS direct outputs)
    static constexpr int LPP = SMAX <= 12 ? 8 : 32;
};

// The batch loop's barrier: the calling thread's group (named barrier 1 + group over C::GT threads).
// bar.sync is the .aligned form, undefined for a warp whose lanes are apart, and code whose trip counts differ from
// lane to lane (rows, direct outputs, large rho^2) runs up to it: the lanes are brought together first.
// (barrier.sync, which needs no convergence, took 53.67 instead of 53.28 ms for 512 images x 9216 sets.)
template <class C>
__device__ __forceinline__ void batch_sync() {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / C::GT), "n"(C::GT) : "memory");
}

// Stage A for one column kx of one pair: Q(dy, kx) for dy = -SMAX..SMAX, with the rows ky = b + R a
// of sub-sequence b transformed by an in-register FFT and recombined with the twiddles
// twc[b][d] = W_N^(b d), d = 0..SMAX, and their conjugates (shared memory, the same address for every
// thread: broadcast).
// The projection column is read from global memory one sub-sequence ahead of its use.  With zcol
// set (the packed edge columns) the inputs are zcol[ky] instead of the product.
template <class C>
__device__ __forceinline__ void stage_a_column(float2 (&acc)[C::NS], const float2* __restrict__ img_col,
                                               const float2* __restrict__ ps_col, const float2* __restrict__ twc,
                                               const float2* __restrict__ zcol, int b0 = 0, int b1 = C::R) {
    constexpr int H = C::H, R = C::R, SMAX = C::SMAX;
    float2 cn[L];
    if constexpr (C::ASPLIT > 1) {
        img_col += b0 * H;
        ps_col += b0 * H;
    }
    if constexpr (C::PREFETCH) {
        if (!zcol) {
#pragma unroll
            for (int a = 0; a < L; ++a) cn[a] = __ldg(ps_col + (R * a) * H);
        }
    }
#pragma unroll 1
    for (int b = b0; b < b1; ++b) {
        float2 x[L];
        if (zcol) {
#pragma unroll
            for (int a = 0; a < L; ++a) x[a] = zcol[R * a + b];
        } else if constexpr (C::PREFETCH) {
#pragma unroll
            for (int a = 0; a < L; ++a) x[a] = c_mulc(img_col[(R * a) * H], cn[a]);
            if (b + 1 < b1) {
#pragma unroll
                for (int a = 0; a < L; ++a) cn[a] = __ldg(ps_col + (R * a + 1) * H);
            }
        } else {
#pragma unroll
            for (int a = 0; a < L; ++a) x[a] = c_mulc(img_col[(R * a) * H], __ldg(ps_col + (R * a) * H));
        }
        img_col += H;
        ps_col += H;
        fft_dif<L>(x);
        // W^(b d) and W^(-b d) are complex conjugates: one twiddle serves dy = +d and -d
        const float2* tw = twc + b * C::TWS;
#pragma unroll
        for (int d = 0; d <= SMAX; ++d) {
            const float2 w = tw[d];
            {
                const int mi = SMAX + d;
                const int u = bitrev(pmod(mi - SMAX, L), ilog2(L));
                acc[mi].x = fmaf(w.x, x[u].x, fmaf(-w.y, x[u].y, acc[mi].x));
                acc[mi].y = fmaf(w.x, x[u].y, fmaf(w.y, x[u].x, acc[mi].y));
            }
            if (d > 0) {
                const int mi = SMAX - d;
                const int u = bitrev(pmod(mi - SMAX, L), ilog2(L));
                acc[mi].x = fmaf(w.x, x[u].x, fmaf(w.y, x[u].y, acc[mi].x));
                acc[mi].y = fmaf(w.x, x[u].y, fmaf(-w.y, x[u].x, acc[mi].y));
            }
        }
    }
}

// Stage B for one row: rho-part(dx) = Re sum_{kx < N/2} w_kx Q(dy, kx) W_N^(kx dx), kx = b + R a;
// only a < L/2 carries data (kx < N/2 for every b < R).  With C::TW2, twc holds 2 W_N^(b d) (the
// weight w = 2 of kx != 0) and the kx = 0 term enters halved; scaling by 2 is exact, so the sums
// are those of the scaled inputs bit for bit.
template <class C>
__device__ __forceinline__ void stage_b_row(float (&acc)[C::NS], const float2* __restrict__ qrow,
                                            const float2* __restrict__ twc, int b0, int b1) {
    constexpr int R = C::R, SMAX = C::SMAX;
#pragma unroll 1
    for (int b = b0; b < b1; ++b) {
        float2 x[L];
#pragma unroll
        for (int a = 0; a < L / 2; ++a) x[a] = C::TW2 ? qrow[b + R * a] : c_scale(qrow[b + R * a], 2.f);
        if (b == 0) x[0] = make_float2((C::TW2 ? 0.5f : 1.f) * qrow[0].x, 0.f);   // kx = 0: weight 1, real
        fft_dif_half_zero<L>(x);
        const float2* tw = twc + b * C::TWS;   // conjugate pairs, as in stage A
#pragma unroll
        for (int d = 0; d <= SMAX; ++d) {
            const float2 w = tw[d];
            {
                const int mi = SMAX + d;
                const int u = bitrev(pmod(mi - SMAX, L), ilog2(L));
                acc[mi] = fmaf(w.x, x[u].x, fmaf(-w.y, x[u].y, acc[mi]));
            }
            if (d > 0) {
                const int mi = SMAX - d;
                const int u = bitrev(pmod(mi - SMAX, L), ilog2(L));
                acc[mi] = fmaf(w.x, x[u].x, fmaf(w.y, x[u].y, acc[mi]));
            }
        }
    }
}

// 2^x by the PTX instruction ex2.approx (relative error about 2^-22; results below 2^-126 flush to
// zero, far below the FP32 resolution of a sum that holds a term equal to 1).  The stage-B sum of
// exp((3 - n)/2 (t - t_min)) takes it with the factor (3 - n)/2 log2(e) folded into one constant:
// one instruction per displacement (6.5 % less k_score time than __expf at 128 px, +-16 px).
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct Part {
    float t;   // min ln(1 - rho^2)
    float s;   // sum exp(c1 (t(d) - t))
    int d;     // index of the minimum, (dy + SMAX) * NS + (dx + SMAX)
};

__device__ __forceinline__ Part merge(Part a, Part b, float c1) {
    if (b.t > a.t || (b.t == a.t && b.d > a.d)) {
        const Part tmp = a;
        a = b;
        b = tmp;
    }
    // now b.t <= a.t (b holds the minimum, lowest index on ties)
    if (!(a.t < INFINITY)) return b;
    Part r;
    r.t = b.t;
    r.d = b.d;
    r.s = b.s + a.s * __expf(c1 * (a.t - b.t));
    return r;
}

// t = ln(1 - rho^2) as ln1m gives it, with |rho| >= 1 (no finite likelihood) flagged in the status
// word and clamped; both tests sit on the rarely taken rho^2 > 1/32 branch.
__device__ __forceinline__ float loglik_t(float rho, int* status) {
    float r2 = rho * rho;
    float t = ln1m_series(r2);
    if (r2 > 0.03125f) {
        if (r2 >= 1.0f) {
            atomicOr(status, BIOEM_DEV_NUMERIC);
            r2 = 1.0f - 5.9604645e-8f;
        }
        t = log1pf(-r2);
    }
    return t;
}

// Shared-memory arrays of a scoring block (pairs j of all groups; group g owns [g GPB, (g + 1) GPB)).
template <class C>
struct Sm {
    float2* img;    // [N][H] the item's image
    float2* q;      // [PB][NS][QS] stage-A output
    float2* twc;    // [R][TWS] twiddles, a second table with C::TW2
    float2* z;      // [PB][N] packed edge columns (C::PACK)
    float* row_t;   // [NGROUP][ROWS] per-row parts
    float* row_s;
    int* row_d;
    float* dir_t;   // [NGROUP][NDIR] the dy = +SMAX row's ln(1 - rho^2)
    float2* dtw;    // [2][R][SMAX + 1] (C::DIRFFT)
    float* dsum;    // [PB][2][SMAX + 1]
    float2* gtw;    // [N] exp(-2 pi i t / N) for the directly evaluated row (C::GTW)
    __device__ __forceinline__ explicit Sm(unsigned char* smem) {
        img = reinterpret_cast<float2*>(smem);
        q = reinterpret_cast<float2*>(smem + C::SM_IMG);
        twc = reinterpret_cast<float2*>(smem + C::SM_IMG + C::SM_QA);
        z = reinterpret_cast<float2*>(smem + C::SM_IMG + C::SM_QA + C::SM_TWC);   // with C::ZALIAS also row_t
        row_t = reinterpret_cast<float*>(smem + C::SM_IMG + C::SM_QA + C::SM_TWC + C::SM_Z);
        row_s = row_t + C::NGROUP * C::ROWS;
        row_d = reinterpret_cast<int*>(row_s + C::NGROUP * C::ROWS);
        dir_t = reinterpret_cast<float*>(row_d + C::NGROUP * C::ROWS);
        dtw = reinterpret_cast<float2*>(smem + C::SM_BASE);
        dsum = reinterpret_cast<float*>(smem + C::SM_BASE + C::SM_DTW);
        gtw = reinterpret_cast<float2*>(smem + C::SM_BASE + C::SM_DTW + C::SM_DSUM);
    }
};

// One work item's operands.  k_score's come from its parameters; where they differ from item to item the
// structure lies in shared memory and is read where it is used (4 models x 4 stacks: 15.94 -> 15.12 ms; kept in
// registers the addresses cost spills, read from the segment table in global memory they wait for the L2).
struct Job {
    const float2* gtw;     // exp(-2 pi i t / N), t < N
    const float2* img;     // the image's spectrum
    const int* ps_idx;     // null, or the list of parameter sets
    const float2* ps;      // parameter-set spectra
    int ps_begin;          // without ps_idx: the wave's first set
    int s;
    float c1;
    float* rec_t;          // the image's record row, indexed by the wave-relative set
    float* rec_s;
    int* rec_d;
};

// Stage B (row transforms), the dy = +SMAX row, the likelihood epilogue and the per-pair combine of
// one batch of the calling group whose Q (stage-A output, [pair][dy][kx]) is in sm.q; records for pairs
// p0 .. hi-1.
// between: what the threads do before the pieces are combined.
template <class C, class F>
__device__ __forceinline__ void score_tail(const Sm<C>& sm, const Job& job, int p0, int hi, int* __restrict__ status,
                                           F&& between) {
    const int s = job.s;
    const float c1 = job.c1;
    constexpr int N = C::N, NC = C::NC, NS = C::NS, SMAX = C::SMAX, NROW = C::NROW, BS = C::BSPLIT;
    const int grp = threadIdx.x / C::GT, tg = threadIdx.x - grp * C::GT;
    // ---------------- stage B: one row (dy = -SMAX .. SMAX-1) of one pair per task (per two
    // adjacent threads with BSPLIT = 2)
#pragma unroll 1
    for (int task = tg; task < C::ROWS; task += C::GT) {
        const int rr = task / BS;
        const int h = task - rr * BS;
        const int jl = rr / NROW;
        const int r = rr - jl * NROW;
        const float2* qrow = sm.q + ((size_t)(grp * C::GPB + jl) * NS + r) * C::QS;
        float acc[NS];
#pragma unroll
        for (int m = 0; m < NS; ++m) acc[m] = 0.f;
        stage_b_row<C>(acc, qrow, sm.twc + (C::TW2 ? C::R * C::TWS : 0), h * (C::R / BS), (h + 1) * (C::R / BS));
        constexpr int MH = BS == 2 ? (NS + 1) / 2 : NS;   // outputs evaluated by this thread
        int m0 = 0;
        if constexpr (BS == 2) {
#pragma unroll
            for (int m = 0; m < NS; ++m) acc[m] += __shfl_xor_sync(0xffffffffu, acc[m], 1);
            // the second thread moves its outputs m = MH .. NS-1 to acc[0 ..]
#pragma unroll
            for (int i = 0; i < MH; ++i) acc[i] = h ? (i + MH < NS ? acc[i + MH] : 0.f) : acc[i];
            m0 = h * MH;
        }
        const float qn = C::PACK ? qrow[0].y : qrow[NC].x;   // Nyquist column, weight 1, phase (-1)^dx
        const bool row_ok = abs(r - SMAX) <= s;
        float tmin = INFINITY;
        int arg = 0x7fffffff;
        // the full window (s = SMAX, uniform over the block) needs no per-output window test
        const float qa = ((m0 - SMAX) & 1) ? -qn : qn;   // the Nyquist term of output i is (-1)^i qa
        const float c1l = c1 * 1.44269504088896341f;
        float ssum = 0.f;
        auto eval = [&](auto full) {
#pragma unroll
            for (int i = 0; i < MH; ++i) {
                const int m = m0 + i;
                const float rho = acc[i] + ((i & 1) ? -qa : qa);
                // full window: every output but the second thread's padding slot (m = NS) counts
                const bool ok = decltype(full)::value ? (i < MH - 1 || m < NS)
                                                      : (row_ok && m < NS && abs(m - SMAX) <= s);
                const float t = ok ? loglik_t(rho, status) : INFINITY;
                acc[i] = t;
                if (t < tmin) {
                    tmin = t;
                    arg = r * NS + m;
                }
            }
            // with the full window t_min is finite, and a left-out output's +inf gives 2^-inf = 0
#pragma unroll
            for (int i = 0; i < MH; ++i) {
                if constexpr (decltype(full)::value)
                    ssum += ex2_approx(c1l * (acc[i] - tmin));
                else
                    ssum += (acc[i] < INFINITY) ? ex2_approx(c1l * (acc[i] - tmin)) : 0.f;
            }
        };
        if (s >= SMAX)
            eval(std::true_type{});
        else
            eval(std::false_type{});
        const int o = grp * C::ROWS + task;
        sm.row_t[o] = tmin;
        sm.row_s[o] = ssum;
        sm.row_d[o] = arg;
    }
    // ---------------- the dy = +SMAX row by real transforms (see Cfg::DIRFFT)
    if constexpr (C::DIRFFT) {
        constexpr int NJG = C::GPB * 2 * C::R;   // jobs: (pair j, component c, sub-sequence b)
        static_assert(C::R == 8 && NJG <= C::GT, "one job per thread");
        // the last NJG threads of the group (the upper half of a warp when that is 16)
        constexpr unsigned JM = NJG >= 32 ? 0xffffffffu : (0xffffffffu << (32 - NJG));   // job lanes
        const int tj = tg - (C::GT - NJG);
        const int b = tj & 7, c = (tj >> 3) & 1, j = grp * C::GPB + (tj >> 4);
        const float2* qrow = sm.q + ((size_t)j * NS + 2 * SMAX) * C::QS;
        if (tj >= 0) {
            float x[8], yr[9], yi[9], a17[SMAX + 1];
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                const float2 v = qrow[b + 8 * a];
                x[a] = c ? v.y : v.x;
            }
            // packed column 0 = (Q(dy, 0), Q(dy, N/2)): weight 1 (the table carries 2), the Nyquist
            // part enters as (-1)^dx Q(dy, N/2) below
            if (b == 0) x[0] = c ? 0.f : 0.5f * x[0];
            rdft16(x, yr, yi);
#pragma unroll
            for (int k = 0; k <= SMAX; ++k) a17[k] = 0.f;
            recombine<SMAX + 1>(a17, yr, yi, sm.dtw + (c * C::R + b) * (SMAX + 1));
#pragma unroll
            for (int k = 0; k <= SMAX; ++k) {
                a17[k] += __shfl_xor_sync(JM, a17[k], 1);
                a17[k] += __shfl_xor_sync(JM, a17[k], 2);
                a17[k] += __shfl_xor_sync(JM, a17[k], 4);
            }
            float* dsum = sm.dsum;
            if (b == 0) {
#pragma unroll
                for (int k = 0; k <= SMAX; ++k) dsum[(j * 2 + c) * (SMAX + 1) + k] = a17[k];
            }
            __syncwarp(JM);
            // lane (c, b) of pair j: dx = b and b + 8 (and 16 for b = 0), sign + for c = 0, - for c = 1
            const float qn = qrow[0].y;
            const bool row_ok = SMAX <= s;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const int dx = r == 0 ? b : (r == 1 ? b + 8 : 2 * 8);
                if ((r == 2 && b != 0) || (c == 1 && dx == 0)) continue;
                const float cv = dsum[(j * 2) * (SMAX + 1) + dx], sv = dsum[(j * 2 + 1) * (SMAX + 1) + dx];
                const float rho = cv + (c ? sv : -sv) + ((dx & 1) ? -qn : qn);
                const int dxs = c ? -dx : dx;
                sm.dir_t[j * NS + dxs + SMAX] = (row_ok && abs(dxs) <= s) ? loglik_t(rho, status) : INFINITY;
            }
        }
    } else {
        // ---------------- the dy = +SMAX row, one output per task, evaluated directly; the threads
        // after the last stage-B row take the first outputs
#pragma unroll 1
        for (int i = (tg + C::GT - C::ROWS % C::GT) % C::GT; i < C::NDIR; i += C::GT) {
            const int jl = i / NS;
            const int mi = i - jl * NS;
            const int dx = mi - SMAX;
            const float2* qrow = sm.q + ((size_t)(grp * C::GPB + jl) * NS + 2 * SMAX) * C::QS;
            float accv = 0.f;
            int idx = pmod(dx, N);
            const int step = idx;
            for (int kx = 1; kx < NC; ++kx) {
                const float2 v = qrow[kx];
                const float2 wv = C::GTW ? sm.gtw[idx] : __ldg(job.gtw + idx);   // exp(-i theta): Re(v exp(+i theta)) = v.x w.x + v.y w.y
                accv = fmaf(v.x, wv.x, fmaf(v.y, wv.y, accv));
                idx += step;
                idx -= (idx >= N) ? N : 0;
            }
            const float qn = C::PACK ? qrow[0].y : qrow[NC].x;
            const float rho = qrow[0].x + 2.f * accv + ((dx & 1) ? -qn : qn);
            const bool ok = SMAX <= s && abs(dx) <= s;
            sm.dir_t[grp * C::NDIR + i] = ok ? loglik_t(rho, status) : INFINITY;
        }
    }
    between();
    batch_sync<C>();
    // ---------------- combine the pieces of each pair: LPP lanes per pair, on the group's first warps
    constexpr int LPP = C::LPP, NR = NROW * BS;
#pragma unroll 1
    for (int e = tg; (e & ~31) < C::GPB * LPP; e += C::GT) {
        const int jl = min(e / LPP, C::GPB - 1), l = e % LPP;
        const float* row_t = sm.row_t + grp * C::ROWS + jl * NR;
        const float* row_s = sm.row_s + grp * C::ROWS + jl * NR;
        const int* row_d = sm.row_d + grp * C::ROWS + jl * NR;
        const float* dir_t = sm.dir_t + grp * C::NDIR + jl * NS;
        Part acc{INFINITY, 0.f, 0x7fffffff};
        for (int r = l; r < NR; r += LPP) acc = merge(acc, Part{row_t[r], row_s[r], row_d[r]}, c1);
        for (int mi = l; mi < NS; mi += LPP) {
            const float t = dir_t[mi];
            acc = merge(acc, Part{t, t < INFINITY ? 1.f : 0.f, 2 * SMAX * NS + mi}, c1);
        }
#pragma unroll
        for (int off = LPP / 2; off > 0; off >>= 1) {
            Part o;
            o.t = __shfl_xor_sync(0xffffffffu, acc.t, off);
            o.s = __shfl_xor_sync(0xffffffffu, acc.s, off);
            o.d = __shfl_xor_sync(0xffffffffu, acc.d, off);
            acc = merge(acc, o, c1);   // merge orders its operands, so both lanes agree
        }
        const int p = p0 + jl;
        // spectra of NaN leave no piece with a value, and which piece wins depends on the lanes: an empty record
        // (ln L = -inf), as 32 lanes with fewer pieces gave
        if (LPP < 32 && !(acc.t < INFINITY)) acc = Part{INFINITY, 0.f, 0x7fffffff};
        if (l == 0 && e < C::GPB * LPP && p < hi) {
            job.rec_t[p] = acc.t;
            job.rec_s[p] = acc.s;
            job.rec_d[p] = acc.d;
        }
    }
}

// The block's constant tables (once per launch; a block barrier follows before their first use).
template <class C>
__device__ __forceinline__ void score_tables(const Sm<C>& sm, const float2* __restrict__ gtw) {
    constexpr int N = C::N, SMAX = C::SMAX;
    const float2* cwN = cw_table<N>();
    for (int i = threadIdx.x; i < C::R * C::TWS; i += C::THREADS) {
        const int b = i / C::TWS, d = i - (i / C::TWS) * C::TWS;
        const float2 w = d <= SMAX ? cwN[pmod(b * d, N)] : make_float2(0.f, 0.f);
        sm.twc[i] = w;
        if constexpr (C::TW2) sm.twc[C::R * C::TWS + i] = make_float2(2.f * w.x, 2.f * w.y);
    }
    if constexpr (C::GTW)
        for (int i = threadIdx.x; i < N; i += C::THREADS) sm.gtw[i] = __ldg(gtw + i);
    if constexpr (C::DIRFFT) {
        // (T1, T2) x 2 (the weight of kx != 0) for component c, sub-sequence b, output dx
        for (int i = threadIdx.x; i < 2 * C::R * (SMAX + 1); i += C::THREADS) {
            const int c = i / (C::R * (SMAX + 1)), b = (i / (SMAX + 1)) % C::R, dx = i % (SMAX + 1);
            const int u = dx & 15;
            const bool cj = u > 8;
            const float2 w = cwN[(b * dx) % N];   // (cos, sin) of 2 pi b dx / N
            const float t1 = c == 0 ? w.x : w.y;
            const float t2 = c == 0 ? (cj ? w.y : -w.y) : (cj ? -w.x : w.x);
            sm.dtw[i] = make_float2(2.f * t1, 2.f * t2);
        }
    }
}

// One work item: the job's image against its parameter sets [lo, hi).
template <class C>
__device__ __forceinline__ void score_item(const Sm<C>& sm, const Job& job, int lo, int hi, int* __restrict__ status) {
    constexpr int N = C::N, NC = C::NC, H = C::H, NS = C::NS, GT = C::GT, GPB = C::GPB;
    __shared__ int next_pair;            // first pair of the item's next untaken batch
    __shared__ int group_next[C::NGROUP];
    const int grp = threadIdx.x / GT, tg = threadIdx.x - grp * GT;
    __syncthreads();   // the previous item's readers of shared memory are done
    {
        const float4* src = reinterpret_cast<const float4*>(job.img);
        float4* dst = reinterpret_cast<float4*>(sm.img);
        for (int i = threadIdx.x; i < N * H / 2; i += C::THREADS) dst[i] = __ldg(src + i);
        if (threadIdx.x == 0) next_pair = lo + C::PB;
    }
    __syncthreads();
    // packed edge columns Z(ky) = P(ky, 0) + i P(ky, N/2) of the batch at p0, by the group's threads
    // first .. first + count - 1
    auto edge_columns = [&](int p0, int first, int count) {
        if (tg < first || tg >= first + count) return;
        for (int i = tg - first; i < GPB * N; i += count) {
            const int jl = i / N;
            const int ky = i - jl * N;
            const int p = min(p0 + jl, hi - 1);
            const int gp = job.ps_idx ? __ldg(job.ps_idx + p) : job.ps_begin + p;
            const float2* ps_row = job.ps + (size_t)gp * N * H + (size_t)ky * H;
            const float2 e0 = c_mulc(sm.img[ky * H], __ldg(ps_row));
            const float2 e1 = c_mulc(sm.img[ky * H + NC], __ldg(ps_row + NC));
            sm.z[grp * GPB * N + i] = make_float2(e0.x - e1.y, e0.y + e1.x);
        }
    };
    if constexpr (C::PACK && !C::ZALIAS) {
        if (lo + grp * GPB < hi) {
            edge_columns(lo + grp * GPB, 0, GT);
            batch_sync<C>();
        }
    }
#pragma unroll 1
    for (int p0 = lo + grp * GPB; p0 < hi;) {
        if constexpr (C::ZALIAS) {
            batch_sync<C>();   // the previous batch's pieces have been combined
            edge_columns(p0, 0, GT);
            batch_sync<C>();
        }
        // ---------------- stage A: one column of one pair per task (per two threads with ASPLIT = 2)
#pragma unroll 1
        for (int e = tg; e < C::TASKS_A * C::ASPLIT; e += GT) {
            const int half = C::ASPLIT == 2 ? e / C::TASKS_A : 0, task = e - half * C::TASKS_A;
            const int jl = task / C::NCOL;
            const int kx = task - jl * C::NCOL;
            const int p = min(p0 + jl, hi - 1);
            const int gp = job.ps_idx ? __ldg(job.ps_idx + p) : job.ps_begin + p;
            const float2* ps_col = job.ps + (size_t)gp * N * H + kx;
            const int j = grp * GPB + jl;
            float2 acc[NS];
#pragma unroll
            for (int m = 0; m < NS; ++m) acc[m] = make_float2(0.f, 0.f);
            constexpr int RS = C::R / C::ASPLIT;
            stage_a_column<C>(acc, sm.img + kx, ps_col, sm.twc, (C::PACK && kx == 0) ? sm.z + j * N : nullptr, half * RS,
                              (half + 1) * RS);
            float2* qdst = sm.q + (size_t)j * NS * C::QS + kx;
            if constexpr (C::ASPLIT == 1) {
#pragma unroll
                for (int m = 0; m < NS; ++m) qdst[m * C::QS] = acc[m];
            } else {
                // each thread stores its sums of one half of the outputs and adds those of the other half to
                // its partner's (one task per thread: every thread of the group passes the barrier once)
                constexpr int MH = (NS + 1) / 2;
#pragma unroll
                for (int m = 0; m < NS; ++m)
                    if ((m < MH) == (half == 0)) qdst[m * C::QS] = acc[m];
                batch_sync<C>();
#pragma unroll
                for (int m = 0; m < NS; ++m)
                    if ((m < MH) != (half == 0)) qdst[m * C::QS] = c_add(qdst[m * C::QS], acc[m]);
            }
        }
        // the group's next batch: written before the barrier, read between it and the next one
        if (tg == 0) group_next[grp] = atomicAdd(&next_pair, GPB);
        batch_sync<C>();
        const int pn = group_next[grp];
        score_tail<C>(sm, job, p0, hi, status, [&]() {
            // the next batch's edge columns by the threads that are free first (Cfg::ZFIRST)
            if constexpr (C::PACK && !C::ZALIAS)
                if (pn < hi) edge_columns(pn, C::ZFIRST, C::ZCOUNT);
        });
        p0 = pn;
    }
}

// Share w of n of `sets` consecutive spectra from src, fetched to the L2 by the lanes of one warp.  The images of a
// chunk go through it side by side, so each of its spectra would be waited for from DRAM by all of them:
// a block fetches its image's share of the chunk that starts half a grid of items later (and, with the
// first items, of its own).  ns per pair without -> with, 64 images: 128 px, +-16 px 12.85 -> 12.1; 192 px, 32 images
// 53 -> 49.2.  A quarter or three quarters of a grid ahead are the same, a whole one is too much for the L2.
template <class C>
__device__ __forceinline__ void fetch_share(const float2* src, int sets, int w, int n) {
    constexpr unsigned kPiece = 4096;
    const long long bytes = (long long)sets * C::N * C::H * (int)sizeof(float2);   // whole 16-byte units
    const long long pieces = (bytes + kPiece - 1) / kPiece;
    for (long long i = pieces * w / n + (threadIdx.x & 31); i < pieces * (w + 1) / n; i += 32) {
        const unsigned len = (unsigned)min((long long)kPiece, bytes - i * kPiece);
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(
                         __cvta_generic_to_global(reinterpret_cast<const char*>(src) + i * kPiece)),
                     "r"(len)
                     : "memory");
    }
}

// Parameter sets of the short chunks that end a launch: a quarter of the others, whole group batches.
template <class C>
__host__ __device__ constexpr int short_chunk(int chunk) {
    return (chunk / 4 + C::GPB - 1) / C::GPB * C::GPB;
}

// Work items (chunk ci, image w), item = ci n_img + w, are taken in index order from a global counter
// (zero at launch): the items in flight stay within one or two chunks of parameter sets, so a chunk
// is read from DRAM about once (a fixed item-per-block assignment let the blocks drift apart over
// thousands of items until several chunks competed for the L2; visiting two chunks per image before
// the next image, to reuse each image, made the two chunks compete the same way).  The first n_long chunks
// hold `chunk` sets, the rest a quarter of that, so that the blocks end closer together.
template <class C>
__global__ void __launch_bounds__(C::THREADS, 1)
k_score(const float2* __restrict__ gtw, const float2* __restrict__ img_spec, int n_img,
        const float2* __restrict__ ps_spec, int ps_begin, int ps_count, int chunk, int n_long, int n_items, int s, float c1,
        float* __restrict__ rec_t, float* __restrict__ rec_s, int* __restrict__ rec_d, int* __restrict__ status,
        int* __restrict__ work, int fetch) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int next_item;
    const Sm<C> sm(smem);
    score_tables<C>(sm, gtw);
    for (;;) {
        if (threadIdx.x == 0) next_item = atomicAdd(work, 1);
        __syncthreads();
        const int item = next_item;   // read by every thread before score_item's first barrier
        if (item >= n_items) break;
        const int ci = item / n_img;
        const int w = item - ci * n_img;
        const int tail = short_chunk<C>(chunk);
        auto first_set = [&](int c) { return c < n_long ? c * chunk : n_long * chunk + (c - n_long) * tail; };
        const int lo = first_set(ci);
        const int hi = min(first_set(ci + 1), ps_count);
        if (fetch && threadIdx.x < 32) {
            const long long nx = (long long)item + gridDim.x / 2;
            if (item < (int)gridDim.x) fetch_share<C>(ps_spec + (size_t)(ps_begin + lo) * C::N * C::H, hi - lo, w, n_img);
            if (nx < n_items) {
                const int cn = (int)(nx / n_img), l2 = first_set(cn);
                fetch_share<C>(ps_spec + (size_t)(ps_begin + l2) * C::N * C::H, min(first_set(cn + 1), ps_count) - l2,
                               (int)(nx - (long long)cn * n_img), n_img);
            }
        }
        const size_t row = (size_t)w * ps_count;
        score_item<C>(sm, Job{gtw, img_spec + (size_t)w * C::N * C::H, nullptr, ps_spec, ps_begin, s, c1, rec_t + row, rec_s + row,
                              rec_d + row},
                      lo, hi, status);
    }
}

// Parts end on whole rounds of a block (NGROUP batches) where an image is one round and there are more
// batches than blocks, or a few rounds and still about a round for every block.
__host__ __device__ inline bool whole_rounds(int n_img, int batches, int groups, int grid) {
    const int rounds = (batches + groups - 1) / groups;
    return (long long)n_img * batches > grid && (rounds == 1 || (rounds < 4 && (long long)n_img * rounds * 8 >= 7ll * grid));
}

// Where a block's part of the work ends within an image of `len` sets (or batches), v of them into it: whole pieces of
// q.  With few rounds per image a piece is what the groups do side by side: part of one takes as long, and a
// block with the ends of two images waits for both.
__device__ __noinline__ int part_end(long long v, int len, int q) {
    if (v <= 0) return 0;
    if (v >= len) return len;
    return min(len, ((int)v + q / 2) / q * q);
}

// The wave's sets go by in phases of phase_sets, whose spectra stay in the L2.  Within a phase the (image, batch)
// pairs, image by image, are split evenly over the blocks, counting a new image as kImageUnits batches
// of a group (its load and the wait of the groups for one another): a block meets one image, or the end of one
// and the start of the next, and every block ends a phase at the same time.
template <class C>
__global__ void __launch_bounds__(C::THREADS, 1)
k_score_phases(const float2* __restrict__ gtw, const float2* __restrict__ img_spec, int n_img,
        const float2* __restrict__ ps_spec, int ps_begin, int ps_count, int phase_sets, int piece, int s, float c1,
        float* __restrict__ rec_t, float* __restrict__ rec_s, int* __restrict__ rec_d, int* __restrict__ status) {
    constexpr int kImageUnits = (6 * C::NGROUP + 5) / 10 > 0 ? (6 * C::NGROUP + 5) / 10 : 1;   // about 0.6 of a round
    extern __shared__ __align__(16) unsigned char smem[];
    const Sm<C> sm(smem);
    score_tables<C>(sm, gtw);
    for (int f0 = 0; f0 < ps_count; f0 += phase_sets) {
        const int f1 = min(f0 + phase_sets, ps_count);
        const int units = (f1 - f0 + C::GPB - 1) / C::GPB, stride = units + kImageUnits;
        const long long all = (long long)n_img * stride;
        // (the blocks' parts shift from phase to phase, so that none always gets two images)
        const int part = (int)((blockIdx.x + 61ll * (f0 / phase_sets)) % gridDim.x);
        const long long x0 = all * part / gridDim.x, x1 = all * (part + 1) / gridDim.x;
        for (int w = (int)(x0 / stride); w < n_img; ++w) {
            const long long at = (long long)w * stride + kImageUnits;   // of the image's first batch
            if (at >= x1) break;
            int u0 = (int)max(x0 - at, 0ll), u1 = (int)min(x1 - at, (long long)units);
            if (piece > 1) {
                u0 = part_end(x0 - at, units, piece);
                u1 = part_end(x1 - at, units, piece);
            }
            if (u0 >= u1) continue;
            const size_t row = (size_t)w * ps_count;
            score_item<C>(sm, Job{gtw, img_spec + (size_t)w * C::N * C::H, nullptr, ps_spec, ps_begin, s, c1, rec_t + row,
                                  rec_s + row, rec_d + row},
                          f0 + u0 * C::GPB, min(f0 + u1 * C::GPB, f1), status);
        }
    }
}

// ---------------------------------------------------------------------------- reductions (float64)
struct Acc {
    double M;    // running max
    double S;    // sum exp(. - M)
    double bv;   // best ln L
    int bp;      // its parameter set
    int bd;      // its displacement index
};

constexpr int kRedThreads = 256;
constexpr int kExpBits = 8;   // table of 2^(j / 256)
__device__ double g_exp2[1 << kExpBits];   // uploaded with the twiddle tables

// exp(x) for x in [-100, 0]: x = (256 q + j) ln2 / 256 + r, |r| <= ln2 / 512, exp(x) = 2^q 2^(j/256) e^r with the
// Taylor series of e^r to r^4 (truncation below 4e-17), the table-driven scheme of Tang (ACM TOMS 15,
// 1989), ln2 / 256 in two float64 numbers (with one the error grows with |x|, to 1.4e-15 at -36).  Within 1.1
// ulp, as the library's exponential is within 1.  Nine float64 operations: the reductions below are bound by the
// float64 pipe (1/70 of the FP32 rate), so what can be an integer operation (comparisons, scaling) is one.
__device__ __forceinline__ double exp_neg(double x, const double* tab) {
    const double big = 6755399441055744.0;   // 1.5 * 2^52: adding it rounds to an integer in the low word
    const double kd = fma(x, 369.32993046757463, big);   // 256 / ln 2
    const int k = __double2loint(kd);
    const double n = kd - big;
    const double r = fma(n, -9.0587766165871077e-20, fma(n, -0.0027076061740622863, x));   // ln 2 / 256
    double p = fma(r, 1.0 / 24.0, 1.0 / 6.0);
    p = fma(r, p, 0.5);
    p = fma(r, p, 1.0);
    const double t = tab[k & ((1 << kExpBits) - 1)];
    const double v = fma(t, r * p, t);
    return __hiloint2double(__double2hiint(v) + (k >> kExpBits) * (1 << 20), __double2loint(v));
}

// Order-preserving integer of a float64 that is not NaN, and back.
__device__ __forceinline__ long long d_key(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double key_d(long long k) { return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll)); }
constexpr long long kKeyNone = (long long)0x800fffffffffffffull;   // -inf

// d > -100 for a difference d <= 0 that is not NaN, by its high word
__device__ __forceinline__ bool in_reach(double d) { return (unsigned)__double2hiint(d) < 0xc0590000u; }

// s exp(d) for d <= 0 that is not NaN; 0 beyond the reach
__device__ __forceinline__ double scaled_exp(double s, double d, const double* tab) {
    return in_reach(d) ? s * exp_neg(d, tab) : 0.0;
}

// Running ln sum = M + ln S; key: of M (kKeyNone: empty).
struct Lse {
    double M = -INFINITY, S = 0.0;
    long long key = kKeyNone;
};

// Folds four terms s_i exp(m_i) (m = -inf or NaN: none) into a; returns the index of the first term that is a
// new maximum, or -1.  Terms more than 100 below the maximum cannot change S (S >= 1: the maximum's own
// s is at least 1) and are left out.
__device__ __forceinline__ int lse_add4(Lse& a, const double (&m)[4], const float (&s)[4], const double* tab) {
    long long k[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        k[i] = d_key(m[i]);
        if ((__double2hiint(m[i]) & 0x7fffffff) >= 0x7ff00000) k[i] = kKeyNone;   // NaN, -inf (+inf does not occur)
    }
    const long long mx = max(max(k[0], k[1]), max(k[2], k[3]));
    int at = -1;
    if (mx > a.key) {
        at = k[0] == mx ? 0 : k[1] == mx ? 1 : k[2] == mx ? 2 : 3;
        const double mv = key_d(mx);
        if (a.key != kKeyNone) a.S = scaled_exp(a.S, a.M - mv, tab);
        a.M = mv;
        a.key = mx;
    }
    if (a.key == kKeyNone) return at;
    bool use[4], any = false;
    double d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        d[i] = m[i] - a.M;
        use[i] = k[i] != kKeyNone && in_reach(d[i]);
        any |= use[i];
    }
    if (any) {
        double e[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) e[i] = exp_neg(use[i] ? d[i] : 0.0, tab);
#pragma unroll
        for (int i = 0; i < 4; ++i) a.S = fma((double)(use[i] ? s[i] : 0.f), e[i], a.S);
    }
    return at;
}

// The table, one entry per thread: loaded before a reduction's first terms, stored after them, so that a small
// call waits once for both.
static_assert((1 << kExpBits) == kRedThreads, "one entry of the table per thread");
__device__ __forceinline__ double exp_entry() { return g_exp2[threadIdx.x]; }

// The warp's sums and best set merged into every lane, lanes in a fixed order; bp = the lowest set of the maximum.
__device__ __forceinline__ void warp_lse(Lse& a, int& bp, const double* tab) {
    long long mx = a.key;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    const double mv = key_d(mx);
    if (a.key != mx) {   // (exp(0) = 1; a small call has few lanes to scale)
        a.S = a.key != kKeyNone ? scaled_exp(a.S, a.M - mv, tab) : 0.0;
        bp = 0x7fffffff;
    }
    a.M = mv;
    a.key = mx;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a.S += __shfl_xor_sync(0xffffffffu, a.S, off);
        bp = min(bp, __shfl_xor_sync(0xffffffffu, bp, off));
    }
}

// The same over a block of kRedThreads, valid in warp 0.
__device__ __forceinline__ void block_lse(Lse& a, int& bp, const double* tab) {
    constexpr int W = kRedThreads / 32;
    __shared__ double rM[W], rS[W];
    __shared__ long long rk[W];
    __shared__ int rb[W];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    warp_lse(a, bp, tab);
    if (lane == 0) { rM[warp] = a.M; rS[warp] = a.S; rk[warp] = a.key; rb[warp] = bp; }
    __syncthreads();
    if (warp == 0) {
        a = Lse{};
        bp = 0x7fffffff;
        if (lane < W) { a.M = rM[lane]; a.S = rS[lane]; a.key = rk[lane]; bp = rb[lane]; }
        warp_lse(a, bp, tab);
    }
}

// r merged with the running accumulator of earlier waves (which hold the lower parameter sets).
__device__ __forceinline__ void acc_merge_prev(Acc& r, const Acc& prev) {
    if (!(prev.M > -INFINITY)) return;
    if (r.M > prev.M) {
        r.S += prev.S * exp(prev.M - r.M);
    } else {
        r.S = r.M > -INFINITY ? prev.S + r.S * exp(r.M - prev.M) : prev.S;
        r.M = prev.M;
    }
    if (prev.bv >= r.bv) { r.bv = prev.bv; r.bp = prev.bp; r.bd = prev.bd; }
}

// One block per (image, part): fold the part's share of the wave's pair records into parts[image][part]
// and, if requested, write the per-orientation posteriors of the share's orientations.  Parts are whole
// orientations; an image is cut into enough of them to occupy the GPU (reduce_parts).  An image in one part
// is folded in place (parts = prev = the running accumulators; prev null: the first wave).  Bound by the
// float64 pipe (14 operations per record; 64 images x 6912 sets: 93 us as one block per image with the
// library's exponential, 33 us so; 16 images with per-orientation output: 181 -> 16 us).
__global__ void __launch_bounds__(kRedThreads) k_reduce_wave(
    const float* __restrict__ rec_t, const float* __restrict__ rec_s, const int* __restrict__ rec_d,
    const double* __restrict__ kA, const double* __restrict__ kB, int ps_begin, int wave_len, int nctf,
    int nq, double c1, double log_norm_orient, Acc* parts, int n_parts, const Acc* prev,
    double* __restrict__ logP_orient) {
    __shared__ double tab[1 << kExpBits];
    const int w = blockIdx.x / n_parts, part = blockIdx.x - w * n_parts;
    const int q_all = wave_len / nctf, q_per = (q_all + n_parts - 1) / n_parts;
    const int q0 = min(part * q_per, q_all), q1 = min(q0 + q_per, q_all);
    const double entry = exp_entry();
    const double ka = kA[w];
    const size_t base = (size_t)w * wave_len;
    Lse a;
    int bp = 0x7fffffff;
    auto term = [&](int p, bool ok, double& m, float& sv) {
        m = ok ? ka + kB[ps_begin + p] + c1 * (double)rec_t[base + p] : -INFINITY;
        sv = ok ? rec_s[base + p] : 0.f;
    };
    double m[4];
    float sv[4];
    if (!logP_orient) {
        const int hi = q1 * nctf;
        int p = q0 * nctf + threadIdx.x;
        auto terms = [&]() {
#pragma unroll
            for (int i = 0; i < 4; ++i) term(p + i * kRedThreads, p + i * kRedThreads < hi, m[i], sv[i]);
        };
        terms();
        tab[threadIdx.x] = entry;
        __syncthreads();
        while (p < hi) {
            const int at = lse_add4(a, m, sv, tab);
            if (at >= 0) bp = p + at * kRedThreads;
            p += 4 * kRedThreads;
            if (p < hi) terms();
        }
    } else {
        tab[threadIdx.x] = entry;
        __syncthreads();
        // an orientation per thread: its sum over the PSFs is an output and one term of the image's sum
        for (int ql = q0 + threadIdx.x; ql < q1; ql += kRedThreads) {
            Lse o;
            int op = 0x7fffffff;
            for (int c = 0; c < nctf; c += 4) {
#pragma unroll
                for (int i = 0; i < 4; ++i) term(ql * nctf + c + i, c + i < nctf, m[i], sv[i]);
                const int at = lse_add4(o, m, sv, tab);
                if (at >= 0) op = ql * nctf + c + at;
            }
            logP_orient[(size_t)w * nq + ps_begin / nctf + ql] = o.M + log(o.S) - log_norm_orient;
            if (o.key > a.key) {
                a.S = a.key != kKeyNone ? o.S + scaled_exp(a.S, a.M - o.M, tab) : o.S;
                a.M = o.M;
                a.key = o.key;
                bp = op;
            } else if (o.key != kKeyNone) {
                a.S += scaled_exp(o.S, o.M - a.M, tab);
            }
        }
    }
    block_lse(a, bp, tab);
    if (threadIdx.x == 0) {
        const bool any = bp != 0x7fffffff;
        Acc r{a.M, a.S, any ? a.M : -INFINITY, any ? ps_begin + bp : 0x7fffffff, any ? rec_d[base + bp] : 0};
        if (prev) acc_merge_prev(r, prev[w]);
        parts[blockIdx.x] = r;
    }
}

// One warp per image: the wave's parts (at most 32, one per lane) and, unless this is the first wave, the
// running accumulator, merged into acc[image]; after the last wave the outputs.  parts null: acc is complete.
__global__ void __launch_bounds__(kRedThreads) k_finalize(Acc* acc, const Acc* parts,
                                                          int n_parts, int first, int last, int n_img, double log_norm,
                                                          int nctf, int nsk, int smax, double* logP, int* best_q,
                                                          int* best_ctf, int* best_dx, int* best_dy, double* best_logL) {
    __shared__ double tab[1 << kExpBits];
    const int w = blockIdx.x * (kRedThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (n_parts > 1) {
        tab[threadIdx.x] = exp_entry();
        __syncthreads();
    }
    if (w >= n_img) return;
    Acc a{-INFINITY, 0.0, -INFINITY, 0x7fffffff, 0};
    if (lane < n_parts) a = (parts ? parts : acc)[(size_t)w * n_parts + lane];
    Acc prev{-INFINITY, 0.0, -INFINITY, 0x7fffffff, 0};
    if (!first) prev = acc[w];
    Lse l;
    if (a.M > -INFINITY) { l.M = a.M; l.S = a.S; l.key = d_key(a.M); }
    int bp = a.bp;
    if (n_parts > 1) warp_lse(l, bp, tab);   // one part: lane 0 has it
    const int src = __ffs(__ballot_sync(0xffffffffu, bp != 0x7fffffff && a.bp == bp)) - 1;
    const int bd = __shfl_sync(0xffffffffu, a.bd, src < 0 ? 0 : src);
    if (lane != 0) return;
    Acc r{l.M, l.S, bp != 0x7fffffff ? l.M : -INFINITY, bp, bd};
    acc_merge_prev(r, prev);
    acc[w] = r;
    if (!last) return;
    if (logP) logP[w] = r.M + log(r.S) - log_norm;
    if (best_q) best_q[w] = r.bp / nctf;
    if (best_ctf) best_ctf[w] = r.bp % nctf;
    if (best_dy) best_dy[w] = r.bd / nsk - smax;
    if (best_dx) best_dx[w] = r.bd % nsk - smax;
    if (best_logL) best_logL[w] = r.bv;
}

// pair_max[w][col0 + p] = max_d ln L and pair_lse[w][col0 + p] = ln sum_d L for the wave's records.
__global__ void k_pairs_out(const float* __restrict__ rec_t, const float* __restrict__ rec_s,
                            const double* __restrict__ kA, const double* __restrict__ kB, int n_img, int ps_begin,
                            int count, double c1, double* pair_max, double* pair_lse, int row_stride, int col0) {
    const size_t total = (size_t)n_img * count;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int w = (int)(i / count);
        const int p = (int)(i - (size_t)w * count);
        const double m = kA[w] + kB[ps_begin + p] + c1 * (double)rec_t[i];
        const size_t o = (size_t)w * row_stride + col0 + p;
        pair_max[o] = m;
        if (pair_lse) pair_lse[o] = m + log((double)rec_s[i]);
    }
}

// Fold this call's per-image (max, sum) into the caller's running pairs acc2[w] = (M, S), ln sum L =
// M + ln S; first != 0 overwrites.
__global__ void k_fold_acc(const Acc* __restrict__ acc, int n_img, double* __restrict__ acc2, int first) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= n_img) return;
    double M = acc[w].M, S = acc[w].S;
    if (!first) {
        const double M0 = acc2[2 * w], S0 = acc2[2 * w + 1];
        if (M0 > -INFINITY) {
            if (!(M > -INFINITY)) { M = M0; S = S0; }
            else if (M0 > M) { S = S * exp(M - M0) + S0; M = M0; }
            else S += S0 * exp(M0 - M);
        }
    }
    acc2[2 * w] = M;
    acc2[2 * w + 1] = S;
}

// ---------------------------------------------------------------------------- host side
// Parts per image of the wave reduction: about four blocks per SM over all images, each of at least 1024
// records (four per thread) and one orientation, at most 32 (one lane each in k_finalize).
int reduce_parts(const bioem_ctx* ctx, int n_img, long long wave, int nctf) {
    long long n = 4ll * ctx->num_sms / n_img;
    if (n > wave / (4 * kRedThreads)) n = wave / (4 * kRedThreads);
    if (n > wave / nctf) n = wave / nctf;
    return (int)(n < 1 ? 1 : n > 32 ? 32 : n);
}

// Accumulators and parts of n_img images in one array: [n_img] accumulators, then with more than one part
// per image [n_img][n_parts].
size_t reduce_bytes(int n_img, int n_parts) {
    return sizeof(Acc) * (size_t)n_img * (n_parts > 1 ? 1 + n_parts : 1);
}

// The reductions of one wave's records into acc (laid out as in reduce_bytes), and after the last wave the
// outputs.
int launch_reduce(bioem_ctx* ctx, const bioem_images* im, const bioem_projset* ps, int max_shift, int smax, int wbegin,
                  int wl, const float* rec_t, const float* rec_s, const int* rec_d, Acc* acc, int n_parts, bool first,
                  bool last, const bioem_score_out& out) {
    const int n_img = im->n_img, nctf = ps->nctf;
    Acc* parts = n_parts > 1 ? acc + n_img : nullptr;
    const double c1 = 0.5 * (3.0 - (double)(im->nx * im->ny));
    const int S = (2 * max_shift + 1) * (2 * max_shift + 1);
    bioem_launch_begin(ctx, KID_REDUCE_WAVE);
    k_reduce_wave<<<n_img * n_parts, kRedThreads, 0, ctx->stream>>>(rec_t, rec_s, rec_d, im->d_kA, ps->d_kB, wbegin, wl,
                                                                    nctf, ps->nq, c1, log((double)nctf * S),
                                                                    parts ? parts : acc, n_parts,
                                                                    parts || first ? nullptr : acc, out.logP_orient);
    bioem_launch_end(ctx, KID_REDUCE_WAVE);
    if (!parts && !last) return bioem_check_cuda(ctx, cudaGetLastError(), "reduction");
    bioem_launch_begin(ctx, KID_FINALIZE);
    k_finalize<<<(n_img + kRedThreads / 32 - 1) / (kRedThreads / 32), kRedThreads, 0, ctx->stream>>>(
        acc, parts, n_parts, first || !parts, last, n_img, log((double)ps->n_ps * S), nctf, 2 * smax + 1, smax, out.logP,
        out.best_q, out.best_ctf, out.best_dx, out.best_dy, out.best_logL);
    bioem_launch_end(ctx, KID_FINALIZE);
    return bioem_check_cuda(ctx, cudaGetLastError(), "reduction");
}

// The wave loop shared by the scoring forms: parameter sets [range) in waves whose per-pair records
// (n_img x wave) fit the scratch limit; `records(wbegin, wl, rec_t, rec_s, rec_d)` enqueues the
// kernel(s) writing the records of sets [wbegin, wbegin + wl), then the float64 reductions fold
// them.  Records name displacements d = (dy + smax) ns + (dx + smax), ns = 2 smax + 1 (smax: the
// record kernel's window, which may exceed the scored max_shift); the posterior is normalised by the
// S = (2 max_shift + 1)^2 scored displacements.  Waves are multiples of `align` parameter sets (whole
// orientations when per-orientation output is wanted).
template <class Records>
int run_waves(bioem_ctx* ctx, const bioem_images* im, const bioem_projset* ps, int max_shift, int smax, int align,
              const bioem_score_out& out, Records&& records) {
    const int n_img = im->n_img;
    const int n = im->nx * im->ny;
    const bool pairs_mode = out.pair_max != nullptr;
    const int range_begin = pairs_mode ? out.ps_begin : 0;
    const int range_len = pairs_mode ? out.ps_count : ps->n_ps;
    const int nctf = ps->nctf;
    if (n_img == 0 || range_len == 0) return BIOEM_OK;

    // wave length: records of n_img x wave must fit the scratch limit; a multiple of `align`
    const unsigned long long per_ps = (unsigned long long)n_img * 12ull;
    long long wave = (long long)(ctx->scratch_limit / per_ps);
    if (wave >= align) wave -= wave % align;
    const long long min_wave = pairs_mode ? 1 : nctf;
    if (wave < min_wave) wave = min_wave;
    if (!pairs_mode) wave -= wave % nctf;
    if (wave > range_len) wave = range_len;
    const size_t rec_need = (size_t)n_img * (size_t)wave * 12;
    if (ctx->rec_bytes < rec_need) {
        if (ctx->d_rec) cudaFreeAsync(ctx->d_rec, ctx->stream);
        ctx->d_rec = nullptr;
        ctx->rec_bytes = 0;
        if (cudaMallocAsync(&ctx->d_rec, rec_need, ctx->stream) != cudaSuccess)
            return bioem_set_error(ctx, BIOEM_ERR_OOM, "record scratch of %zu bytes", rec_need);
        ctx->rec_bytes = rec_need;
    }
    const int n_parts = pairs_mode ? 1 : reduce_parts(ctx, n_img, wave, nctf);
    // for the most parts that n_img images are ever cut into: a call captured in a graph must find the
    // accumulators in place, whatever number of sets the earlier calls of as many images had
    const size_t acc_need = sizeof(Acc) * ((size_t)n_img + 4 * (size_t)ctx->num_sms);
    if (!pairs_mode && ctx->acc_bytes < acc_need) {
        if (ctx->d_acc) cudaFreeAsync(ctx->d_acc, ctx->stream);
        ctx->d_acc = nullptr;
        ctx->acc_bytes = 0;
        if (cudaMallocAsync(&ctx->d_acc, acc_need, ctx->stream) != cudaSuccess)
            return bioem_set_error(ctx, BIOEM_ERR_OOM, "accumulator scratch");
        ctx->acc_bytes = acc_need;
    }
    float* rec_t = reinterpret_cast<float*>(ctx->d_rec);
    float* rec_s = rec_t + (size_t)n_img * wave;
    int* rec_d = reinterpret_cast<int*>(rec_s + (size_t)n_img * wave);
    const double c1 = 0.5 * (3.0 - (double)n);
    Acc* acc = reinterpret_cast<Acc*>(ctx->d_acc);

    for (long long w0 = 0; w0 < range_len; w0 += wave) {
        const int wl = (int)(range_len - w0 < wave ? range_len - w0 : wave);
        const int wbegin = range_begin + (int)w0;
        int rc = records(wbegin, wl, rec_t, rec_s, rec_d);
        if (rc) return rc;
        if (pairs_mode) {
            bioem_launch_begin(ctx, KID_PAIRS_OUT);
            k_pairs_out<<<1024, 256, 0, ctx->stream>>>(rec_t, rec_s, im->d_kA, ps->d_kB, n_img, wbegin, wl, c1,
                                                       out.pair_max, out.pair_lse, range_len, (int)w0);
            bioem_launch_end(ctx, KID_PAIRS_OUT);
        } else {
            rc = launch_reduce(ctx, im, ps, max_shift, smax, wbegin, wl, rec_t, rec_s, rec_d, acc, n_parts,
                               w0 == 0, w0 + wl == range_len, out);
        }
        if (!rc) rc = bioem_check_cuda(ctx, cudaGetLastError(), "reduction");
        if (rc) return rc;
    }
    if (!pairs_mode) {
        if (out.acc2) {
            bioem_launch_begin(ctx, KID_FINALIZE);
            k_fold_acc<<<(n_img + 255) / 256, 256, 0, ctx->stream>>>(acc, n_img, out.acc2, out.acc_first);
            bioem_launch_end(ctx, KID_FINALIZE);
        }
        return bioem_check_cuda(ctx, cudaGetLastError(), "k_fold_acc");
    }
    return BIOEM_OK;
}

// Resident blocks of k_score<C> on the whole GPU (sets the kernel's shared-memory attribute).
template <class C>
int score_slots(bioem_ctx* ctx, int* slots) {
    const size_t smem = C::SMEM;
    const void* kernel;
    if constexpr (C::PHASES) kernel = (const void*)k_score_phases<C>;
    else kernel = (const void*)k_score<C>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return bioem_set_error(ctx, BIOEM_ERR_CUDA, "shared memory attribute (%zu bytes)", smem);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, C::THREADS, smem) != cudaSuccess || per_sm < 1)
        return bioem_set_error(ctx, BIOEM_ERR_CUDA, "occupancy query");
    *slots = per_sm * ctx->num_sms;
    return BIOEM_OK;
}

// Parameter sets per chunk with which the chunks in flight (those of the resident blocks, the one being finished
// and the one being fetched) stay in the L2.
long long l2_sets(long long spec_bytes, int n_img, int slots) {
    return (long long)((48 << 20) / (((double)slots / n_img + 1.5) * (double)spec_bytes));
}

// Parameter sets per work item.  A block's groups take an item's batches from its counter and wait for one
// another between items (about 0.6 of a round of all groups); with more items than slots the last items
// end unevenly (about 0.75 of an item).  Of the even splits of the wl sets into k chunks that the L2 holds (but
// at least eight rounds), the one with the least rounds + waits; measured at 64 images x 4608 sets, 128 px, +-16 px
// (ns per pair): chunks of 123: 12.3, 185: 12.15, 246: 12.2, 512: 12.2.
template <class C>
int score_chunk(int n_img, int wl, int slots) {
    long long cap = l2_sets((long long)sizeof(float2) * C::N * C::H, n_img, slots);
    if (cap < 8 * C::PB) cap = 8 * C::PB;
    const long long k0 = (wl + cap - 1) / cap;
    long long best = (cap + C::GPB - 1) / C::GPB * C::GPB;
    double best_cost = 1e300;
    for (long long k = k0, step = 1; k < 64 * k0 && k <= wl; k += step, step = 1 + k / 16) {
        const long long chunk = ((wl + k - 1) / k + C::GPB - 1) / C::GPB * C::GPB;
        const long long items = (wl + chunk - 1) / chunk * n_img;
        const double turns = items <= slots ? 1.0 : (double)items / slots + 0.75;
        const double cost = turns * ((double)chunk / C::PB + 0.6);
        if (cost < best_cost) {
            best_cost = cost;
            best = chunk;
        }
    }
    return (int)best;
}

// Parameter sets of a phase: 48 MB of spectra, which the L2 keeps (it is two halves, and what one reads from the
// other's memory it holds too: 128 px, s = 4, ns per pair: 24 MB 7.07, 32: 7.04, 48: 6.92, 64: 7.26, 96: 7.71),
// but at least eight rounds of every block.
template <class C>
int phase_sets(int n_img, int wl, int slots) {
    constexpr long long spec = (long long)sizeof(float2) * C::N * C::H;
    long long fit = (48ll << 20) / spec;
    const long long least = (8ll * C::PB * slots + n_img - 1) / n_img;
    if (fit < least) fit = least;
    const long long phases = (wl + fit - 1) / fit;
    return (int)(((wl + phases - 1) / phases + C::GPB - 1) / C::GPB * C::GPB);
}

// One k_score<C> launch writing the records of parameter sets [wbegin, wbegin + wl) for every image.
template <class C>
int launch_score_records(bioem_ctx* ctx, const bioem_images* im, const bioem_projset* ps, int slots, int wbegin,
                         int wl, int max_shift, float* rec_t, float* rec_s, int* rec_d) {
    const int n_img = im->n_img;
    const float c1f = 0.5f * (3.0f - (float)(C::N * C::N));
    if constexpr (C::PHASES) {
        const int phase = phase_sets<C>(n_img, wl, slots);
        const int per_img = ((phase < wl ? phase : wl) + C::GPB - 1) / C::GPB;
        const long long units = (long long)n_img * per_img;
        const int grid = (int)(units < slots ? units : slots);
        const int piece = whole_rounds(n_img, per_img, C::NGROUP, grid) ? C::NGROUP : 1;
        bioem_launch_begin(ctx, KID_SCORE);
        k_score_phases<C><<<grid, C::THREADS, C::SMEM, ctx->stream>>>(bioem_twiddles(ctx, C::N), im->d_spec, n_img, ps->d_spec,
                                                                wbegin, wl, phase, piece, max_shift, c1f, rec_t, rec_s, rec_d,
                                                                ctx->d_status);
        bioem_launch_end(ctx, KID_SCORE);
    } else {
        const long long chunk = score_chunk<C>(n_img, wl, slots);
        // with more items than slots, about the last item of each slot goes out in short chunks: 13.19 -> 12.94 ns
        // per pair at 128 px, +-16 px, 64 images (two or three items' worth gained no more)
        long long n_chunks = (wl + chunk - 1) / chunk, n_long = n_chunks;
        if (n_chunks * n_img > slots && chunk >= 4 * C::GPB) {
            n_long = wl / chunk - ((long long)slots + n_img - 1) / n_img;
            if (n_long < 0) n_long = 0;
            const int tail = short_chunk<C>((int)chunk);
            n_chunks = n_long + (wl - n_long * chunk + tail - 1) / tail;
        }
        const long long n_items = n_chunks * n_img;
        if (n_items > 0x7fffffffll) return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE, "too many work items");
        const int grid = (int)(n_items < slots ? n_items : slots);
        // no fetching ahead in a single round, where it repeats what the blocks are reading, nor where half a grid of
        // items, n_img of which share a chunk, reaches further than the L2 keeps (192 px, 6912 sets, us with
        // and without: 1 image 528 and 466, 2: 899 and 850, 3: 1259 and 1203, 5 (48 MB ahead): 1937 and 1931; 128 px,
        // +-16 px: 1: 217 and 172, 3: 411 and 399, 8 (53 MB): 882 and 917)
        const double ahead = 0.5 * grid / n_img * (double)chunk * (double)(sizeof(float2) * C::N * C::H);
        const int fetch = n_items > slots && ahead < 60e6;
        bioem_launch_begin(ctx, KID_SCORE);
        if (cudaMemsetAsync(ctx->d_work, 0, sizeof(int), ctx->stream) != cudaSuccess)
            return bioem_check_cuda(ctx, cudaGetLastError(), "work counter");
        k_score<C><<<grid, C::THREADS, C::SMEM, ctx->stream>>>(bioem_twiddles(ctx, C::N), im->d_spec, n_img, ps->d_spec,
                                                                wbegin, wl, (int)chunk, (int)n_long, (int)n_items, max_shift, c1f,
                                                                rec_t, rec_s, rec_d, ctx->d_status, ctx->d_work, fetch);
        bioem_launch_end(ctx, KID_SCORE);
    }
    return bioem_check_cuda(ctx, cudaGetLastError(), "k_score");
}

// The FP32 form: k_score<C> writes the records (displacements named in C's compile-time window).
template <class C>
int run_score(bioem_ctx* ctx, const bioem_images* im, const bioem_projset* ps, int max_shift,
              const bioem_score_out& out) {
    int slots = 0;
    const int rc = score_slots<C>(ctx, &slots);
    if (rc) return rc;
    auto records = [&](int wbegin, int wl, float* rec_t, float* rec_s, int* rec_d) -> int {
        return launch_score_records<C>(ctx, im, ps, slots, wbegin, wl, max_shift, rec_t, rec_s, rec_d);
    };
    return run_waves(ctx, im, ps, max_shift, C::SMAX, ps->nctf, out, records);
}

// The split-precision tensor-core form (gemm.cu writes the records, window = max_shift); waves are
// whole 128-set row tiles where the scratch allows.
int run_score_gemm(bioem_ctx* ctx, const bioem_images* im, const bioem_projset* ps, int max_shift,
                   const bioem_score_out& out) {
    const int mode = ctx->precision;
    int rc = bioem_gemm_prepare(ctx, im, ps, max_shift, mode);
    if (rc) return rc;
    const int tile = bioem_gemm_row_tile();
    int a = tile, b = ps->nctf;
    while (b) { const int t = a % b; a = b; b = t; }
    const int align = tile / a * ps->nctf;   // lcm(row tile, PSFs per orientation)
    auto records = [&](int wbegin, int wl, float* rec_t, float* rec_s, int* rec_d) -> int {
        return bioem_gemm_records(ctx, im, ps, max_shift, mode, wbegin, wbegin + wl, rec_t, rec_s, rec_d);
    };
    return run_waves(ctx, im, ps, max_shift, max_shift, align, out, records);
}

// <N, SMAX, groups, threads per group, pairs per group batch, packed edge columns[, threads per
// stage-B row]>.  Groups as many as registers allow without spills and shared memory holds; a group's batch
// fills whole rounds of its threads with column tasks (PB N/2 with the packed edge columns, PB (N/2 + 1)
// without) and at most one round with rows.  ns per pair (k_score, one GB300; one block-wide group of
// 245-272 threads moving through the phases in step before -> now): 32 px 1.76 -> 0.78; 64 px, s = 4: 3.68 ->
// 2.07, s = 8: 5.22 -> 2.90; 96 px 10.5 -> 6.85; 128 px, s = 4: 14.7 -> 6.55.  More groups at fewer registers lost
// (128 px, s = 4: 6 x 128 threads of 79 registers 9.9; 8 x 64 threads 10.4), as did fewer, larger ones
// (3 x 192 threads 7.9, 3 x 256 10.0).  192 px holds two pairs beside the image: one group in step, 49
// (as two groups of one pair 64: the 97th column then takes a warp per group; the image read through L1 and
// three pairs in 10 or 12 warps: 62-73).  The odd column kx = N/2
// stays a column task: spread over a warp's lanes (transforms, then outputs) it took fewer
// instructions but made that warp the batch's longest (64 px, s = 4: 2.4; 96 px 8.6; 192 px 62).
// Packed edge columns where they measured faster (128 px: 2 % at s = 4, 6 % at s = 16); at 32-96 px the
// transforms are short enough that forming Z costs about as much as the column it saves.
using C32_4 = Cfg<32, 4, 6, 128, 15, false>;
using C64_4 = Cfg<64, 4, 5, 128, 11, false>;
using C64_8 = Cfg<64, 8, 3, 160, 9, false>;
using C96_12 = Cfg<96, 12, 3, 128, 5, false>;
using C128_4 = Cfg<128, 4, 4, 160, 5, true>;
using C128_16 = Cfg<128, 16, 4, 128, 2, true, 2>;
using C192_24 = Cfg<192, 24, 1, 224, 2, false>;
// The batched call's 192 px instance (its matrix is FP32): two threads per column and per row, packed edge
// columns: 12 warps instead of 7 on the two pairs that shared memory holds, 54 -> 47 ns per pair.  k_score keeps
// C192_24, whose sums have the order of every other FP32 instance.
using B192_24 = Cfg<192, 24, 1, 384, 2, true, 2, 2>;

}  // namespace

int bioem_score_supported(int npix, int max_shift) {
    if (max_shift < 0 || 2 * max_shift >= npix) return 0;
    switch (npix) {
        case 32: return max_shift <= 4;
        case 64: return max_shift <= 8;
        case 96: return max_shift <= 12;
        case 128: return max_shift <= 16;
        case 192: return max_shift <= 24;
        default: return 0;
    }
}

int bioem_launch_score(bioem_ctx* ctx, const bioem_images* im, const bioem_projset* ps, int max_shift,
                       const bioem_score_out& out) {
    if (ctx->precision == BIOEM_PRECISION_FP16X2_FFT) {
        if (!bioem_tc_supported(im->nx, max_shift))
            return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE,
                                   "tensor-core column transforms: 128 px and max_shift <= 16 only (%d px, %d)",
                                   im->nx, max_shift);
        auto records = [&](int wbegin, int wl, float* rec_t, float* rec_s, int* rec_d) -> int {
            return bioem_tc_records(ctx, im, ps, max_shift, wbegin, wl, rec_t, rec_s, rec_d);
        };
        return run_waves(ctx, im, ps, max_shift, 16, ps->nctf, out, records);
    }
    if (ctx->precision != BIOEM_PRECISION_FP32) {
        if (!bioem_gemm_supported(im->nx, max_shift))
            return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE,
                                   "split-precision form: max_shift %d at %d px exceeds 256 columns per image", max_shift,
                                   im->nx);
        return run_score_gemm(ctx, im, ps, max_shift, out);
    }
    switch (im->nx) {
        case 32: return run_score<C32_4>(ctx, im, ps, max_shift, out);
        case 64: return max_shift <= 4 ? run_score<C64_4>(ctx, im, ps, max_shift, out)
                                       : run_score<C64_8>(ctx, im, ps, max_shift, out);
        case 96: return run_score<C96_12>(ctx, im, ps, max_shift, out);
        case 128: return max_shift <= 4 ? run_score<C128_4>(ctx, im, ps, max_shift, out)
                                        : run_score<C128_16>(ctx, im, ps, max_shift, out);
        case 192: return run_score<C192_24>(ctx, im, ps, max_shift, out);
        default: return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE, "unsupported image size %d", im->nx);
    }
}

int bioem_upload_score_twiddles(bioem_ctx* ctx) {
    const int sizes[6] = {16, 32, 64, 96, 128, 192};
    for (int k = 0; k < 6; ++k) {
        const int M = sizes[k];
        float2 h[192];
        for (int t = 0; t < M; ++t) {
            const double a = 2.0 * 3.14159265358979323846 * (double)t / (double)M;
            h[t] = make_float2((float)cos(a), (float)sin(a));
        }
        cudaError_t e;
        switch (M) {
            case 16: e = cudaMemcpyToSymbol(c_w16, h, sizeof(float2) * 16); break;
            case 32: e = cudaMemcpyToSymbol(c_w32, h, sizeof(float2) * 32); break;
            case 64: e = cudaMemcpyToSymbol(c_w64, h, sizeof(float2) * 64); break;
            case 96: e = cudaMemcpyToSymbol(c_w96, h, sizeof(float2) * 96); break;
            case 192: e = cudaMemcpyToSymbol(c_w192, h, sizeof(float2) * 192); break;
            default: e = cudaMemcpyToSymbol(c_w128, h, sizeof(float2) * 128); break;
        }
        if (e != cudaSuccess) return bioem_check_cuda(ctx, e, "twiddle upload");
    }
    double t[1 << kExpBits];
    for (int j = 0; j < (1 << kExpBits); ++j) t[j] = exp2((double)j / (1 << kExpBits));
    return bioem_check_cuda(ctx, cudaMemcpyToSymbol(g_exp2, t, sizeof(t)), "exponential table upload");
}

// ---------------------------------------------------------------------------- allocation-free scoring
// Scratch for bioem_score_noalloc: per-image accumulators followed by per-pair records, reserved
// statically in device memory on every GPU this library is loaded on, for the life of the process.
// Host code must not use the symbol's host-side address: each device's address is looked up once
// with cudaGetSymbolAddress while that device is current.

namespace {

constexpr size_t kNoAllocBytes = 16u << 20;   // 16 MiB
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
void* g_noalloc_ptr[kMaxDevices] = {};

// Device address of the static scratch on the current device.  Looked up again on every call made
// outside a stream capture (a device reset between calls reloads the module, possibly at another
// address); a call made while the stream is capturing uses the address of the last such lookup.
int noalloc_scratch(bioem_ctx* ctx, void** out) {
    if (ctx->device < 0 || ctx->device >= kMaxDevices)
        return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE, "device ordinal %d too large", ctx->device);
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(ctx->stream, &cs) != cudaSuccess) {
        cudaGetLastError();
        cs = cudaStreamCaptureStatusActive;   // unknown: do not call into the runtime's module table
    }
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (cs == cudaStreamCaptureStatusNone) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) return bioem_check_cuda(ctx, e != cudaSuccess ? e : cudaErrorInvalidSymbol,
                                                             "cudaGetSymbolAddress(static scoring scratch)");
        g_noalloc_ptr[ctx->device] = p;
    } else if (!g_noalloc_ptr[ctx->device]) {
        return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG,
                               "allocation-free scoring: the first call on a device must come before any stream capture");
    }
    *out = g_noalloc_ptr[ctx->device];
    return BIOEM_OK;
}

// The wave loop of bioem_score (log P only) with records and accumulators in the static scratch.
template <class C>
int run_score_noalloc(bioem_ctx* ctx, const bioem_images* im, const bioem_projset* ps, int max_shift, double* logP) {
    const int n_img = im->n_img;
    const int nctf = ps->nctf;
    if (n_img == 0) return BIOEM_OK;
    const size_t acc_bytes = ((sizeof(Acc) * (size_t)n_img + 255) / 256) * 256;
    const size_t per_ps = (size_t)n_img * 12;
    if (acc_bytes + per_ps * nctf > kNoAllocBytes)
        return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE,
                               "allocation-free scoring: %d images x %d PSFs need %zu bytes of scratch, more than "
                               "the static %zu", n_img, nctf, acc_bytes + per_ps * nctf, kNoAllocBytes);
    void* base = nullptr;
    int rc = noalloc_scratch(ctx, &base);
    if (rc) return rc;
    // the reduction's parts follow the accumulators where they leave the records room
    int n_parts = reduce_parts(ctx, n_img, ps->n_ps, nctf);
    size_t head = (reduce_bytes(n_img, n_parts) + 255) / 256 * 256;
    if (head + per_ps * nctf > kNoAllocBytes) {
        n_parts = 1;
        head = acc_bytes;
    }
    long long wave = (long long)((kNoAllocBytes - head) / per_ps);
    wave -= wave % nctf;
    if (wave > ps->n_ps) wave = ps->n_ps;
    Acc* acc = reinterpret_cast<Acc*>(base);
    float* rec_t = reinterpret_cast<float*>(static_cast<unsigned char*>(base) + head);
    float* rec_s = rec_t + (size_t)n_img * wave;
    int* rec_d = reinterpret_cast<int*>(rec_s + (size_t)n_img * wave);

    int slots = 0;
    rc = score_slots<C>(ctx, &slots);
    if (rc) return rc;
    bioem_score_out out{};
    out.logP = logP;
    for (long long w0 = 0; w0 < ps->n_ps; w0 += wave) {
        const int wl = (int)(ps->n_ps - w0 < wave ? ps->n_ps - w0 : wave);
        rc = launch_score_records<C>(ctx, im, ps, slots, (int)w0, wl, max_shift, rec_t, rec_s, rec_d);
        if (!rc)
            rc = launch_reduce(ctx, im, ps, max_shift, C::SMAX, (int)w0, wl, rec_t, rec_s, rec_d, acc, n_parts, w0 == 0,
                               w0 + wl == ps->n_ps, out);
        if (rc) return rc;
    }
    return BIOEM_OK;
}

}  // namespace

extern "C" int bioem_score_noalloc(bioem_ctx* ctx, const bioem_images* images, const bioem_projset* projset,
                                   int max_shift, double* d_logP) {
    if (!ctx || !images || !projset) return BIOEM_ERR_INVALID_ARG;
    if (images->ctx != ctx || projset->ctx != ctx)
        return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "handle from another context");
    if (images->nx != projset->nx || images->ny != projset->ny ||
        fabs(images->pixel_A - projset->pixel_A) > 1e-9 * images->pixel_A)
        return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "images and projections differ in size or pixel");
    if (max_shift < 0) return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "negative max_shift");
    if (!bioem_score_supported(images->nx, max_shift))
        return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE, "max_shift %d unsupported at %d px", max_shift,
                               images->nx);
    if (projset->n_ps == 0) return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "empty parameter set");
    if (images->n_img > 0 && !d_logP) return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "d_logP is required");
    if (cudaSetDevice(ctx->device) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "cudaSetDevice");
    switch (images->nx) {
        case 32: return run_score_noalloc<C32_4>(ctx, images, projset, max_shift, d_logP);
        case 64: return max_shift <= 4 ? run_score_noalloc<C64_4>(ctx, images, projset, max_shift, d_logP)
                                       : run_score_noalloc<C64_8>(ctx, images, projset, max_shift, d_logP);
        case 96: return run_score_noalloc<C96_12>(ctx, images, projset, max_shift, d_logP);
        case 128: return max_shift <= 4 ? run_score_noalloc<C128_4>(ctx, images, projset, max_shift, d_logP)
                                        : run_score_noalloc<C128_16>(ctx, images, projset, max_shift, d_logP);
        case 192: return run_score_noalloc<C192_24>(ctx, images, projset, max_shift, d_logP);
        default: return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE, "unsupported image size %d", images->nx);
    }
}

// ---------------------------------------------------------------------------- batched scoring
// Several models against several image stacks of mixed sizes.  A segment is one (model, stack) pair:
// the stack's image spectra against that model's parameter sets for that stack.  The segments of one
// image size form one work list, run by one persistent launch of that size's scoring instance; the
// launches of the sizes present are parallel branches of the graph, so that the blocks of the next
// size start on the SMs that the previous size's blocks leave.  (One kernel that held all four sizes
// gave every size the register count and the 256 threads of the largest: 19.2 ms for 4 models x 4
// stacks, 1.03e6 pairs; 16.1 ms by size, 13.9 with the instances' other changes.)
#include <string>
#include <vector>

namespace {

struct SegDesc {
    const float2* img;    // [n_img][N][N/2+1]
    const float2* ps;     // [n_ps][N][N/2+1]
    const float2* gtw;    // exp(-2 pi i t / N)
    const double* kA;     // [n_img]
    const double* kB;     // [n_ps]
    float* rec_t;         // [n_img][n_ps] records
    float* rec_s;
    int* rec_d;
    long long item_begin; // first item of this segment among those of its image size
    long long row_begin;  // first global reduction row (image) of this segment
    int n_img, n_ps, chunk, n_chunks, s, npix, nctf;
    int out_row;          // model index (row of the output matrix)
    int out_col;          // column of the segment's first image in the output matrix
    float c1;
    double log_norm;      // ln(n_ps S)
};

__device__ __forceinline__ int find_seg(const SegDesc* segs, int n, long long x, bool rows) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        const long long b = rows ? segs[mid].row_begin : segs[mid].item_begin;
        if (b <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Work items of the segments of one image size, in index order from a global counter (zero at launch),
// as in k_score.
template <class C>
__global__ void __launch_bounds__(C::THREADS, 1)
k_score_segs(const SegDesc* __restrict__ segs, int n_segs, long long n_items, int* __restrict__ status,
             unsigned long long* __restrict__ work) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long next_item;
    __shared__ Job job;
    const Sm<C> sm(smem);
    score_tables<C>(sm, segs[0].gtw);   // the same for every segment: one image size
    for (;;) {
        if (threadIdx.x == 0) next_item = (long long)atomicAdd(work, 1ull);
        __syncthreads();
        const long long item = next_item;
        if (item >= n_items) break;
        const int g = find_seg(segs, n_segs, item, false);
        const SegDesc& sd = segs[g];
        const long long local = item - sd.item_begin;
        const int ci = (int)(local / sd.n_img);
        const int w = (int)(local - (long long)ci * sd.n_img);
        const int lo = ci * sd.chunk;
        const int hi = min(lo + sd.chunk, sd.n_ps);
        if (threadIdx.x < 32) {
            if (item < (long long)gridDim.x) fetch_share<C>(sd.ps + (size_t)lo * C::N * C::H, hi - lo, w, sd.n_img);
            const long long nx = item + gridDim.x / 2;
            if (nx < n_items) {
                const SegDesc& sn = segs[find_seg(segs, n_segs, nx, false)];
                const long long k = nx - sn.item_begin;
                const int cn = (int)(k / sn.n_img), l2 = cn * sn.chunk;
                fetch_share<C>(sn.ps + (size_t)l2 * C::N * C::H, min(l2 + sn.chunk, sn.n_ps) - l2, (int)(k - (long long)cn * sn.n_img),
                               sn.n_img);
            }
        }
        const size_t row = (size_t)w * sd.n_ps;
        if (threadIdx.x == 0)   // the previous item's readers are past the barrier above
            job = Job{sd.gtw, sd.img + (size_t)w * C::N * C::H, nullptr, sd.ps, 0, sd.s, sd.c1, sd.rec_t + row, sd.rec_s + row,
                      sd.rec_d + row};
        __syncthreads();
        score_item<C>(sm, job, lo, hi, status);
    }
}

using SegKernel = void (*)(const SegDesc*, int, long long, int*, unsigned long long*);
struct SegInstance {
    SegKernel kernel;
    int threads, smem, smax;
    int unit;   // chunk sizes are multiples of this (the unit that tune files have always used)
};

// The instance that scores the segments of an image size (null kernel: not a batched size).
SegInstance seg_instance(int npix) {
    switch (npix) {
        case 64: return {k_score_segs<C64_8>, C64_8::THREADS, (int)C64_8::SMEM, C64_8::SMAX, 15};
        case 96: return {k_score_segs<C96_12>, C96_12::THREADS, (int)C96_12::SMEM, C96_12::SMAX, 10};
        case 128: return {k_score_segs<C128_16>, C128_16::THREADS, (int)C128_16::SMEM, C128_16::SMAX, 7};
        case 192: return {k_score_segs<B192_24>, B192_24::THREADS, (int)B192_24::SMEM, B192_24::SMAX, 2};
        default: return {nullptr, 0, 0, 0, 1};
    }
}

// Resident blocks of the instance on the whole GPU (sets the kernel's shared-memory attribute).
int seg_slots(bioem_ctx* ctx, const SegInstance& si, int* slots) {
    if (cudaFuncSetAttribute(si.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, si.smem) != cudaSuccess)
        return bioem_set_error(ctx, BIOEM_ERR_CUDA, "shared memory attribute (%d bytes)", si.smem);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, si.kernel, si.threads, si.smem) != cudaSuccess || per_sm < 1)
        return bioem_set_error(ctx, BIOEM_ERR_CUDA, "occupancy query");
    *slots = per_sm * ctx->num_sms;
    return BIOEM_OK;
}

// One block per (segment, image): float64 log-sum-exp over the image's records, written as float32
// into out[model][column].
__global__ void __launch_bounds__(kRedThreads) k_reduce_multi(const SegDesc* __restrict__ segs, int n_segs,
                                                              float* __restrict__ out, int out_ld) {
    __shared__ double tab[1 << kExpBits];
    const double entry = exp_entry();
    const long long row = blockIdx.x;
    const int g = find_seg(segs, n_segs, row, true);
    const SegDesc& sd = segs[g];
    const int w = (int)(row - sd.row_begin);
    const double ka = sd.kA[w];
    const double c1 = (double)sd.c1;
    Lse a;
    int bp = 0x7fffffff;
    const size_t base = (size_t)w * sd.n_ps;
    double m[4];
    float sv[4];
    int p = threadIdx.x;
    auto terms = [&]() {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int pi = p + i * kRedThreads;
            m[i] = pi < sd.n_ps ? ka + sd.kB[pi] + c1 * (double)sd.rec_t[base + pi] : -INFINITY;
            sv[i] = pi < sd.n_ps ? sd.rec_s[base + pi] : 0.f;
        }
    };
    terms();
    tab[threadIdx.x] = entry;
    __syncthreads();
    while (p < sd.n_ps) {
        lse_add4(a, m, sv, tab);
        p += 4 * kRedThreads;
        if (p < sd.n_ps) terms();
    }
    block_lse(a, bp, tab);
    if (threadIdx.x == 0)
        out[(size_t)sd.out_row * out_ld + sd.out_col + w] = (float)(a.M + log(a.S) - sd.log_norm);
}

struct TuneEntry {
    int npix, s, chunk;
};

int default_chunk(int npix) { return npix >= 192 ? 64 : 256; }   // at most

int tuned_chunk(const std::vector<TuneEntry>& t, int npix, int s) {
    for (const auto& e : t)
        if (e.npix == npix && e.s == s) return e.chunk;
    return 0;
}

// Without an entry: the default, halved while the L2 does not hold the chunks in flight (4 models x 4 stacks of 16
// to 32 images: 14.95 -> 13.8 ms).
int untuned_chunk(int npix, int n_img, int slots) {
    const long long fit = l2_sets((long long)sizeof(float2) * npix * (npix / 2 + 1), n_img, slots);
    int chunk = default_chunk(npix);
    for (int k = 0; k < 2 && chunk > fit; ++k) chunk /= 2;
    return chunk;
}

}  // namespace

struct bioem_batch {
    bioem_ctx* ctx;
    int device;            // bioem_batch_free uses these, never the (possibly destroyed) context
    cudaStream_t stream;
    int n_models, n_stacks, n_cols;
    std::vector<SegDesc> segs;
    SegDesc* d_segs;
    void* d_rec;
    unsigned long long* d_work;   // work-item counters of the scoring launches, one per size
    long long n_rows;
    float* d_out;
    // the segments [seg0, seg0 + n_segs) of one image size and their launch
    struct Group {
        int npix, seg0, n_segs;
        long long n_items;
    };
    std::vector<Group> groups;
    cudaStream_t cap_stream;
    std::vector<cudaStream_t> side;   // capture only: one branch per further size
    std::vector<cudaEvent_t> events;
    cudaGraph_t graph;
    cudaGraphExec_t exec;
};

// tune table kept per process (per image size and shift window)
static std::mutex g_tune_mutex;
static std::vector<TuneEntry> g_tune;

// An entry the batched launch can use: a batched image size, a shift window its instance covers,
// and a chunk that is a whole number of that size's tuning units, at most 4096 parameter sets.
static bool tune_entry_valid(int npix, int s, int chunk) {
    const SegInstance si = seg_instance(npix);
    if (!si.kernel || s < 0 || s > si.smax || 2 * s >= npix) return false;
    return chunk > 0 && chunk <= 4096 && chunk % si.unit == 0;
}

// Read "npix shift chunk" lines into the process table.  Lines that are not three integers, or
// whose entry is not valid, are skipped (a corrupted or foreign cache file then only costs a new
// tuning run); returns the number of entries taken (-1 if the file cannot be opened) and, in
// *skipped, the number of non-blank lines skipped.
static int tune_load(const char* path, int* skipped = nullptr) {
    if (skipped) *skipped = 0;
    FILE* f = fopen(path, "r");
    if (!f) return -1;
    char line[256];
    int n = 0;
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    while (fgets(line, sizeof line, f)) {
        int npix, s, chunk;
        char extra;
        const int got = sscanf(line, "%d %d %d %c", &npix, &s, &chunk, &extra);
        if (got != 3 || !tune_entry_valid(npix, s, chunk)) {
            bool blank = true;
            for (const char* c = line; *c; ++c)
                if (*c != ' ' && *c != '\t' && *c != '\n' && *c != '\r') blank = false;
            if (!blank && skipped) ++*skipped;
            continue;
        }
        bool found = false;
        for (auto& e : g_tune)
            if (e.npix == npix && e.s == s) { e.chunk = chunk; found = true; }
        if (!found) g_tune.push_back({npix, s, chunk});
        ++n;
    }
    fclose(f);
    return n;
}

static int batch_build(bioem_batch* b) {
    bioem_ctx* ctx = b->ctx;
    const size_t nb = sizeof(SegDesc) * b->segs.size(), n_groups = b->groups.size();
    if (cudaMalloc((void**)&b->d_segs, nb) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_OOM, "segment table");
    if (cudaMemcpy(b->d_segs, b->segs.data(), nb, cudaMemcpyHostToDevice) != cudaSuccess)
        return bioem_set_error(ctx, BIOEM_ERR_CUDA, "segment table upload");
    if (cudaMalloc((void**)&b->d_work, sizeof(unsigned long long) * n_groups) != cudaSuccess)
        return bioem_set_error(ctx, BIOEM_ERR_OOM, "work counters");
    std::vector<int> grids(n_groups);
    for (size_t g = 0; g < n_groups; ++g) {
        int slots = 0;
        const int rc = seg_slots(ctx, seg_instance(b->groups[g].npix), &slots);
        if (rc) return rc;
        grids[g] = (int)(b->groups[g].n_items < slots ? b->groups[g].n_items : slots);
    }
    if (cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking) != cudaSuccess)
        return bioem_set_error(ctx, BIOEM_ERR_CUDA, "capture stream");
    for (size_t g = 0; g < n_groups; ++g) {   // one side stream per further size; fork and join events
        cudaStream_t st = nullptr;
        cudaEvent_t ev = nullptr;
        if (g > 0 && cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess)
            return bioem_set_error(ctx, BIOEM_ERR_CUDA, "capture stream");
        if (st) b->side.push_back(st);
        if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess)
            return bioem_set_error(ctx, BIOEM_ERR_CUDA, "capture event");
        b->events.push_back(ev);
    }
    if (cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
        return bioem_set_error(ctx, BIOEM_ERR_CUDA, "begin capture");
    cudaMemsetAsync(b->d_work, 0, sizeof(unsigned long long) * n_groups, b->cap_stream);
    cudaEventRecord(b->events[0], b->cap_stream);
    for (size_t g = 0; g < n_groups; ++g) {
        const bioem_batch::Group& gr = b->groups[g];
        const SegInstance si = seg_instance(gr.npix);
        cudaStream_t st = g == 0 ? b->cap_stream : b->side[g - 1];
        if (g > 0) cudaStreamWaitEvent(st, b->events[0], 0);
        si.kernel<<<grids[g], si.threads, si.smem, st>>>(b->d_segs + gr.seg0, gr.n_segs, gr.n_items, ctx->d_status,
                                                         b->d_work + g);
        if (g > 0) {
            cudaEventRecord(b->events[g], st);
            cudaStreamWaitEvent(b->cap_stream, b->events[g], 0);
        }
    }
    k_reduce_multi<<<(unsigned)b->n_rows, kRedThreads, 0, b->cap_stream>>>(b->d_segs, (int)b->segs.size(), b->d_out,
                                                                           b->n_cols);
    cudaError_t e = cudaStreamEndCapture(b->cap_stream, &b->graph);
    if (e != cudaSuccess) return bioem_check_cuda(ctx, e, "end capture");
    e = cudaGraphInstantiate(&b->exec, b->graph, 0);
    if (e != cudaSuccess) return bioem_check_cuda(ctx, e, "graph instantiate");
    return BIOEM_OK;
}

extern "C" {

int bioem_autotune_load(const char* cache_path, int* n_taken, int* n_skipped) {
    if (!cache_path) return BIOEM_ERR_INVALID_ARG;
    int skipped = 0;
    const int n = tune_load(cache_path, &skipped);
    if (n_taken) *n_taken = n < 0 ? 0 : n;
    if (n_skipped) *n_skipped = skipped;
    return n < 0 ? BIOEM_ERR_INVALID_ARG : BIOEM_OK;
}

int bioem_autotune(bioem_ctx* ctx, const bioem_images* images, const bioem_projset* projset, int max_shift,
                   const char* cache_path, int* out_chunk) {
    if (!ctx || !images || !projset) return BIOEM_ERR_INVALID_ARG;
    if (cache_path && tune_load(cache_path) > 0) {
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        for (const auto& e : g_tune)
            if (e.npix == images->nx && e.s == max_shift) {
                if (out_chunk) *out_chunk = e.chunk;
                return BIOEM_OK;
            }
    }
    const int npix = images->nx;
    const SegInstance si = seg_instance(npix);
    if (!si.kernel)
        return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE, "autotune: batched sizes are 64, 96, 128, 192");
    if (max_shift < 0 || max_shift > si.smax || images->nx != projset->nx || images->n_img == 0 ||
        projset->n_ps == 0)
        return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "autotune: bad case");
    if (cudaSetDevice(ctx->device) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "cudaSetDevice");
    // trial: the first images (up to 2 per SM) against up to 4096 parameter sets, one segment
    const int n_img = images->n_img < 2 * ctx->num_sms ? images->n_img : 2 * ctx->num_sms;
    const int n_ps = projset->n_ps < 4096 ? projset->n_ps : 4096;
    const int pb = si.unit;
    const int cands[5] = {pb * 2, pb * 8, pb * 32, pb * 64, pb * 128};
    int slots = 0;
    const int src = seg_slots(ctx, si, &slots);
    if (src) return src;
    void* rec = nullptr;
    const size_t rec_bytes = (size_t)n_img * n_ps * 12;
    if (cudaMalloc(&rec, rec_bytes) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_OOM, "autotune records");
    double best_ms = 1e300;
    int best = default_chunk(npix);
    int rc = BIOEM_OK;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    for (int k = 0; k < 5 && rc == BIOEM_OK; ++k) {
        const int chunk = cands[k];
        if (chunk > 2 * n_ps && k > 0) break;
        SegDesc sd{};
        sd.img = images->d_spec;
        sd.ps = projset->d_spec;
        sd.gtw = bioem_twiddles(ctx, npix);
        sd.kA = images->d_kA;
        sd.kB = projset->d_kB;
        sd.rec_t = static_cast<float*>(rec);
        sd.rec_s = sd.rec_t + (size_t)n_img * n_ps;
        sd.rec_d = reinterpret_cast<int*>(sd.rec_s + (size_t)n_img * n_ps);
        sd.n_img = n_img;
        sd.n_ps = n_ps;
        sd.chunk = chunk;
        sd.n_chunks = (n_ps + chunk - 1) / chunk;
        sd.s = max_shift;
        sd.npix = npix;
        sd.nctf = projset->nctf;
        sd.c1 = 0.5f * (3.0f - (float)(npix * npix));
        sd.log_norm = 0.0;
        const long long n_items = (long long)sd.n_chunks * n_img;
        SegDesc* d_seg = nullptr;
        if (cudaMalloc((void**)&d_seg, sizeof(SegDesc)) != cudaSuccess) { rc = BIOEM_ERR_OOM; break; }
        cudaMemcpy(d_seg, &sd, sizeof(SegDesc), cudaMemcpyHostToDevice);
        const int grid = (int)(n_items < slots ? n_items : slots);
        double ms_best_rep = 1e300;
        for (int rep = 0; rep < 3; ++rep) {
            cudaEventRecord(e0, ctx->stream);
            cudaMemsetAsync(ctx->d_work, 0, sizeof(unsigned long long), ctx->stream);
            si.kernel<<<grid, si.threads, si.smem, ctx->stream>>>(d_seg, 1, n_items, ctx->d_status,
                                                                  reinterpret_cast<unsigned long long*>(ctx->d_work));
            cudaEventRecord(e1, ctx->stream);
            if (cudaEventSynchronize(e1) != cudaSuccess) { rc = bioem_check_cuda(ctx, cudaGetLastError(), "autotune"); break; }
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep > 0 && ms < ms_best_rep) ms_best_rep = ms;   // first repetition warms up
        }
        cudaFree(d_seg);
        if (ms_best_rep < best_ms) {
            best_ms = ms_best_rep;
            best = chunk;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(rec);
    if (rc) return rc;
    {
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        bool found = false;
        for (auto& e : g_tune)
            if (e.npix == npix && e.s == max_shift) { e.chunk = best; found = true; }
        if (!found) g_tune.push_back({npix, max_shift, best});
        if (cache_path) {
            FILE* f = fopen(cache_path, "w");
            if (f) {
                for (const auto& e : g_tune) fprintf(f, "%d %d %d\n", e.npix, e.s, e.chunk);
                fclose(f);
            }
        }
    }
    if (out_chunk) *out_chunk = best;
    return BIOEM_OK;
}

int bioem_batch_create(bioem_ctx* ctx, int n_models, int n_stacks, const bioem_images* const* stacks,
                       const bioem_projset* const* projsets, const int* max_shift, float* d_logP_matrix,
                       bioem_batch** out) {
    if (!ctx || !out || n_models <= 0 || n_stacks <= 0 || !stacks || !projsets || !max_shift || !d_logP_matrix)
        return BIOEM_ERR_INVALID_ARG;
    *out = nullptr;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "cudaSetDevice");
    bioem_batch* b = new (std::nothrow) bioem_batch();
    if (!b) return BIOEM_ERR_OOM;
    b->ctx = ctx;
    b->device = ctx->device;
    b->stream = ctx->stream;
    b->n_models = n_models;
    b->n_stacks = n_stacks;
    b->d_out = d_logP_matrix;
    int col = 0;
    size_t rec_total = 0;
    std::vector<int> cols(n_stacks);
    for (int k = 0; k < n_stacks; ++k) {
        const bioem_images* im = stacks[k];
        if (!im || im->ctx != ctx) { delete b; return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "stack %d", k); }
        const int npix = im->nx;
        const SegInstance si = seg_instance(npix);
        if (!si.kernel || max_shift[k] < 0 || max_shift[k] > si.smax || 2 * max_shift[k] >= npix) {
            delete b;
            return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE, "stack %d: %d px, shift %d", k, npix, max_shift[k]);
        }
        cols[k] = col;
        col += im->n_img;
    }
    b->n_cols = col;
    for (int m = 0; m < n_models; ++m) {   // every handle is checked before any segment is made
        for (int k = 0; k < n_stacks; ++k) {
            const bioem_images* im = stacks[k];
            const bioem_projset* ps = projsets[(size_t)m * n_stacks + k];
            if (!ps || ps->ctx != ctx || ps->nx != im->nx || fabs(ps->pixel_A - im->pixel_A) > 1e-9 * im->pixel_A ||
                ps->n_ps == 0) {
                delete b;
                return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "projection set (%d, %d) does not match", m, k);
            }
        }
    }
    // segments by image size, the longest items first (the largest images)
    long long rows = 0;
    const int sizes[4] = {192, 128, 96, 64};
    for (int npix : sizes) {
        bioem_batch::Group gr{npix, (int)b->segs.size(), 0, 0};
        for (int mk = 0; mk < n_models * n_stacks; ++mk) {
            const int m = mk / n_stacks, k = mk - m * n_stacks;
            const bioem_images* im = stacks[k];
            const bioem_projset* ps = projsets[mk];
            if (im->nx != npix || im->n_img == 0) continue;
            SegDesc sd{};
            sd.img = im->d_spec;
            sd.ps = ps->d_spec;
            sd.gtw = bioem_twiddles(ctx, im->nx);
            sd.kA = im->d_kA;
            sd.kB = ps->d_kB;
            sd.n_img = im->n_img;
            sd.n_ps = ps->n_ps;
            {
                std::lock_guard<std::mutex> lock(g_tune_mutex);
                sd.chunk = tuned_chunk(g_tune, im->nx, max_shift[k]);
            }
            if (sd.chunk == 0) sd.chunk = untuned_chunk(im->nx, im->n_img, ctx->num_sms);
            sd.n_chunks = (sd.n_ps + sd.chunk - 1) / sd.chunk;
            sd.s = max_shift[k];
            sd.npix = im->nx;
            sd.nctf = ps->nctf;
            sd.out_row = m;
            sd.out_col = cols[k];
            sd.c1 = 0.5f * (3.0f - (float)(im->nx * im->nx));
            const int S = (2 * max_shift[k] + 1) * (2 * max_shift[k] + 1);
            sd.log_norm = log((double)ps->n_ps * S);
            sd.item_begin = gr.n_items;
            sd.row_begin = rows;
            gr.n_items += (long long)sd.n_chunks * sd.n_img;
            rows += sd.n_img;
            rec_total += (size_t)sd.n_img * sd.n_ps * 12;
            b->segs.push_back(sd);
        }
        gr.n_segs = (int)b->segs.size() - gr.seg0;
        if (gr.n_segs) b->groups.push_back(gr);
    }
    b->n_rows = rows;
    if (b->segs.empty()) { delete b; return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "no images"); }
    if (rows > 0x7fffffffll) { delete b; return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE, "too many rows"); }
    if (cudaMalloc(&b->d_rec, rec_total) != cudaSuccess) {
        delete b;
        return bioem_set_error(ctx, BIOEM_ERR_OOM, "batch records of %zu bytes", rec_total);
    }
    size_t off = 0;
    for (auto& sd : b->segs) {
        const size_t npair = (size_t)sd.n_img * sd.n_ps;
        float* base = reinterpret_cast<float*>(static_cast<unsigned char*>(b->d_rec) + off);
        sd.rec_t = base;
        sd.rec_s = base + npair;
        sd.rec_d = reinterpret_cast<int*>(base + 2 * npair);
        off += npair * 12;
    }
    const int rc = batch_build(b);
    if (rc) {
        bioem_batch_free(b);
        return rc;
    }
    *out = b;
    return BIOEM_OK;
}

int bioem_batch_run(bioem_batch* b) {
    if (!b) return BIOEM_ERR_INVALID_ARG;
    bioem_ctx* ctx = b->ctx;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "cudaSetDevice");
    ctx->n_launches += b->groups.size() + 1;
    ctx->kid_launches[KID_SCORE] += b->groups.size();
    ctx->kid_launches[KID_REDUCE_WAVE] += 1;
    return bioem_check_cuda(ctx, cudaGraphLaunch(b->exec, ctx->stream), "graph launch");
}

long long bioem_batch_evals(const bioem_batch* b) {
    if (!b) return -1;
    long long e = 0;
    for (const auto& sd : b->segs) e += (long long)sd.n_img * sd.n_ps;
    return e;
}

void bioem_batch_free(bioem_batch* b) {
    if (!b) return;
    cudaSetDevice(b->device);
    cudaStreamSynchronize(b->stream);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
    for (cudaStream_t st : b->side) cudaStreamDestroy(st);
    for (cudaEvent_t ev : b->events) cudaEventDestroy(ev);
    if (b->d_segs) cudaFree(b->d_segs);
    if (b->d_rec) cudaFree(b->d_rec);
    if (b->d_work) cudaFree(b->d_work);
    cudaGetLastError();
    delete b;
}

}  // extern "C"

// ---------------------------------------------------------------------------- gathered scoring
// Each image against its own list of parameter sets (CSR: offsets[n_img + 1], ps_idx[nnz] into the
// projection set), folded into running per-image float64 (max, sum) accumulators.
namespace {

// The lists, end to end, are split evenly over the blocks, counting an image as kImageSets more sets (its load
// and the wait of the groups for one another, 0.6 of a round); parts end on whole group batches of their
// image's list.  k_score us, items of one image from a counter -> so: 64 images of 512 sets, 128 px, s = 4: 320 ->
// 260; 300 images of 173 sets, 64 px: 214 -> 176; 1024 images of 225 sets, 128 px, s = 16: 2.95 ms either way.
template <class C>
__global__ void __launch_bounds__(C::THREADS, 1)
k_score_gathered(const float2* __restrict__ gtw, const float2* __restrict__ img_spec, int n_img,
                 const int* __restrict__ offsets, const int* __restrict__ ps_idx, const float2* __restrict__ ps_spec, int s,
                 float c1, float* __restrict__ rec_t, float* __restrict__ rec_s, int* __restrict__ rec_d,
                 int* __restrict__ status) {
    constexpr int kImageSets = (6 * C::PB + 5) / 10, GPB = C::GPB;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ Job job;
    __shared__ long long x0, x1;   // the block's part
    __shared__ int next_w, part_lo, part_hi;
    const Sm<C> sm(smem);
    score_tables<C>(sm, gtw);
    auto start = [&](int w) { return (long long)(offsets[w] - offsets[0]) + (long long)w * kImageSets; };
    if (threadIdx.x == 0) {
        const long long all = start(n_img);
        x0 = all * blockIdx.x / gridDim.x;
        x1 = all * (blockIdx.x + 1) / gridDim.x;
        int w = 0;   // the last image that starts at or before x0
        for (int hi = n_img - 1; w < hi;) {
            const int mid = (w + hi + 1) >> 1;
            if (start(mid) <= x0) w = mid;
            else hi = mid - 1;
        }
        next_w = w;
    }
    const bool many = offsets[n_img] - offsets[0] > (long long)gridDim.x * GPB;
    for (;;) {
        __syncthreads();   // the previous image's readers of the job are done
        if (threadIdx.x == 0) {
            part_lo = part_hi = 0;
            for (int w = next_w; w < n_img; ++w) {
                const long long at = start(w) + kImageSets;   // of the image's first set
                if (at >= x1) break;
                const int b0 = offsets[w], len = offsets[w + 1] - b0;
                const int rounds = (len + C::PB - 1) / C::PB;
                const bool whole = many && (rounds == 1 || (rounds < 4 && (long long)n_img * rounds * 8 >= 7ll * gridDim.x));
                const int piece = whole ? C::PB : GPB;
                const int lo = part_end(x0 - at, len, piece), hi = part_end(x1 - at, len, piece);
                if (lo >= hi) continue;
                job = Job{gtw, img_spec + (size_t)w * C::N * C::H, ps_idx + b0, ps_spec, 0, s, c1, rec_t + b0, rec_s + b0,
                          rec_d + b0};
                part_lo = lo;
                part_hi = hi;
                next_w = w + 1;
                break;
            }
        }
        __syncthreads();
        const int lo = part_lo, hi = part_hi;
        if (lo >= hi) break;
        score_item<C>(sm, job, lo, hi, status);
    }
}

__global__ void __launch_bounds__(kRedThreads) k_fold_gathered(const int* __restrict__ offsets,
                                                               const int* __restrict__ ps_idx,
                                                               const float* __restrict__ rec_t,
                                                               const float* __restrict__ rec_s,
                                                               const double* __restrict__ kA,
                                                               const double* __restrict__ kB, double c1,
                                                               double* __restrict__ acc, int first) {
    __shared__ double tab[1 << kExpBits];
    const int w = blockIdx.x;
    const double entry = exp_entry();
    const int b0 = offsets[w], b1 = offsets[w + 1];
    Lse a;
    int bp = 0x7fffffff;
    double m[4];
    float sv[4];
    int i0 = b0 + threadIdx.x;
    auto terms = [&]() {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = i0 + k * kRedThreads;
            m[k] = i < b1 ? kA[w] + kB[ps_idx[i]] + c1 * (double)rec_t[i] : -INFINITY;
            sv[k] = i < b1 ? rec_s[i] : 0.f;
        }
    };
    terms();
    tab[threadIdx.x] = entry;
    __syncthreads();
    while (i0 < b1) {
        lse_add4(a, m, sv, tab);
        i0 += 4 * kRedThreads;
        if (i0 < b1) terms();
    }
    block_lse(a, bp, tab);
    if (threadIdx.x == 0) {
        Acc r{a.M, a.S, -INFINITY, 0, 0};
        if (!first) acc_merge_prev(r, Acc{acc[2 * w], acc[2 * w + 1], -INFINITY, 0, 0});
        acc[2 * w] = r.M;
        acc[2 * w + 1] = r.S;
    }
}

__global__ void k_acc_logP(const double* __restrict__ acc, int n_img, double log_norm, double* __restrict__ logP) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w < n_img) logP[w] = acc[2 * w] + log(acc[2 * w + 1]) - log_norm;
}

// Eq. 9's sum over disjoint parts of a grid: out[w] = the (M, S) pair of the union of the n_parts
// accumulators parts[k][w] (each ln sum L = M + ln S; an empty part has M = -inf), folded in index
// order k = 0, 1, ... so the result does not depend on the launch.  out may be parts (part 0).
__global__ void k_acc_merge(const double* __restrict__ parts, int n_parts, int n, double* out) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= n) return;
    double M = -INFINITY, S = 0.0;
    for (int k = 0; k < n_parts; ++k) {
        const double m2 = parts[((size_t)k * n + w) * 2], s2 = parts[((size_t)k * n + w) * 2 + 1];
        if (!(m2 > -INFINITY)) continue;
        if (m2 > M) { S = S * exp(M - m2) + s2; M = m2; }
        else S += s2 * exp(m2 - M);
    }
    out[2 * w] = M;
    out[2 * w + 1] = S;
}

// out[g] = ln sum_j exp(v[g len + j]) for consecutive groups of len values (a sum of Eq. 9 over a
// few grid points, e.g. the B-factors of one orientation and defocus), max-shifted in float64.
__global__ void k_group_lse(const double* __restrict__ v, long long n_groups, int len, double* __restrict__ out) {
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < n_groups;
         g += (long long)gridDim.x * blockDim.x) {
        const double* x = v + g * len;
        double m = -INFINITY;
        for (int j = 0; j < len; ++j) m = fmax(m, x[j]);
        if (!(m > -INFINITY)) {
            out[g] = m;
            continue;
        }
        double s = 0.0;
        for (int j = 0; j < len; ++j) s += exp(x[j] - m);
        out[g] = m + log(s);
    }
}

// Per listed pair i of image w: ln sum_d L(w | ps_idx[i], d) = kA + kB + c1 t_min + ln s (one block per image).
__global__ void __launch_bounds__(kRedThreads) k_gathered_pairs_out(const int* __restrict__ offsets,
                                                                    const int* __restrict__ ps_idx,
                                                                    const float* __restrict__ rec_t,
                                                                    const float* __restrict__ rec_s,
                                                                    const double* __restrict__ kA,
                                                                    const double* __restrict__ kB, double c1,
                                                                    double* __restrict__ pair_lse) {
    const int w = blockIdx.x;
    const int b0 = offsets[w], b1 = offsets[w + 1];
    for (int i = b0 + threadIdx.x; i < b1; i += blockDim.x)
        pair_lse[i] = kA[w] + kB[ps_idx[i]] + c1 * (double)rec_t[i] + log((double)rec_s[i]);
}

template <class C>
int run_gathered(bioem_ctx* ctx, const bioem_images* im, const bioem_projset* ps, int max_shift, const int* offsets,
                 const int* ps_idx, int nnz, double* acc, int first, double* pair_lse) {
    const int n_img = im->n_img;
    const size_t need = (size_t)nnz * 12;
    if (ctx->rec_bytes < need) {
        if (ctx->d_rec) cudaFreeAsync(ctx->d_rec, ctx->stream);
        ctx->d_rec = nullptr;
        ctx->rec_bytes = 0;
        if (cudaMallocAsync(&ctx->d_rec, need, ctx->stream) != cudaSuccess)
            return bioem_set_error(ctx, BIOEM_ERR_OOM, "record scratch of %zu bytes", need);
        ctx->rec_bytes = need;
    }
    float* rec_t = reinterpret_cast<float*>(ctx->d_rec);
    float* rec_s = rec_t + nnz;
    int* rec_d = reinterpret_cast<int*>(rec_s + nnz);
    const size_t smem = C::SMEM;
    if (cudaFuncSetAttribute(k_score_gathered<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return bioem_set_error(ctx, BIOEM_ERR_CUDA, "shared memory attribute");
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_score_gathered<C>, C::THREADS, smem);
    if (per_sm < 1) per_sm = 1;
    const int slots = per_sm * ctx->num_sms;
    const long long batches = (long long)n_img + nnz / C::GPB;   // at least as many as there are
    const int grid = nnz > 0 ? (int)(batches < slots ? batches : slots) : 0;
    const int n = C::N * C::N;
    if (grid > 0) {
        bioem_launch_begin(ctx, KID_SCORE);
        k_score_gathered<C><<<grid, C::THREADS, smem, ctx->stream>>>(bioem_twiddles(ctx, C::N), im->d_spec, n_img, offsets,
                                                                     ps_idx, ps->d_spec, max_shift,
                                                                     0.5f * (3.0f - (float)n), rec_t, rec_s, rec_d,
                                                                     ctx->d_status);
        bioem_launch_end(ctx, KID_SCORE);
        int rc = bioem_check_cuda(ctx, cudaGetLastError(), "k_score_gathered");
        if (rc) return rc;
    }
    bioem_launch_begin(ctx, KID_REDUCE_WAVE);
    if (pair_lse)
        k_gathered_pairs_out<<<n_img, kRedThreads, 0, ctx->stream>>>(offsets, ps_idx, rec_t, rec_s, im->d_kA, ps->d_kB,
                                                                    0.5 * (3.0 - (double)n), pair_lse);
    else
        k_fold_gathered<<<n_img, kRedThreads, 0, ctx->stream>>>(offsets, ps_idx, rec_t, rec_s, im->d_kA, ps->d_kB,
                                                               0.5 * (3.0 - (double)n), acc, first);
    bioem_launch_end(ctx, KID_REDUCE_WAVE);
    return bioem_check_cuda(ctx, cudaGetLastError(), "k_fold_gathered");
}

}  // namespace

extern "C" {

static int gathered(bioem_ctx* ctx, const bioem_images* images, const bioem_projset* projset, int max_shift,
                    const int* d_offsets, const int* d_ps_idx, int nnz, int max_per_image, double* d_acc, int first,
                    double* d_pair_lse) {
    if (!ctx || !images || !projset || !d_offsets || (!d_acc && !d_pair_lse) || nnz < 0 || max_per_image < 0 ||
        (nnz > 0 && !d_ps_idx))
        return BIOEM_ERR_INVALID_ARG;
    if (images->ctx != ctx || projset->ctx != ctx || images->nx != projset->nx)
        return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "images and projections do not match");
    if (!bioem_score_supported(images->nx, max_shift))
        return bioem_set_error(ctx, BIOEM_ERR_UNSUPPORTED_SIZE, "max_shift %d unsupported at %d px", max_shift,
                               images->nx);
    if (images->n_img == 0) return BIOEM_OK;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "cudaSetDevice");
#define G(C) run_gathered<C>(ctx, images, projset, max_shift, d_offsets, d_ps_idx, nnz, d_acc, first, d_pair_lse)
    switch (images->nx) {
        case 32: return G(C32_4);
        case 64: return max_shift <= 4 ? G(C64_4) : G(C64_8);
        case 96: return G(C96_12);
        case 128: return max_shift <= 4 ? G(C128_4) : G(C128_16);
        default: return G(C192_24);
    }
#undef G
}

int bioem_score_gathered(bioem_ctx* ctx, const bioem_images* images, const bioem_projset* projset, int max_shift,
                         const int* d_offsets, const int* d_ps_idx, int nnz, int max_per_image, double* d_acc,
                         int first) {
    if (!d_acc) return BIOEM_ERR_INVALID_ARG;
    return gathered(ctx, images, projset, max_shift, d_offsets, d_ps_idx, nnz, max_per_image, d_acc, first, nullptr);
}

int bioem_score_gathered_pairs(bioem_ctx* ctx, const bioem_images* images, const bioem_projset* projset, int max_shift,
                               const int* d_offsets, const int* d_ps_idx, int nnz, int max_per_image,
                               double* d_pair_lse) {
    if (!d_pair_lse && nnz > 0) return BIOEM_ERR_INVALID_ARG;
    if (nnz == 0) return BIOEM_OK;
    return gathered(ctx, images, projset, max_shift, d_offsets, d_ps_idx, nnz, max_per_image, nullptr, 0, d_pair_lse);
}

int bioem_acc_merge(bioem_ctx* ctx, const double* d_parts, int n_parts, int n, double* d_out) {
    if (!ctx || n_parts < 1 || n < 0 || (n > 0 && (!d_parts || !d_out))) return BIOEM_ERR_INVALID_ARG;
    if (n == 0) return BIOEM_OK;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "cudaSetDevice");
    bioem_launch_begin(ctx, KID_LSE_MERGE);
    k_acc_merge<<<(n + 255) / 256, 256, 0, ctx->stream>>>(d_parts, n_parts, n, d_out);
    bioem_launch_end(ctx, KID_LSE_MERGE);
    return bioem_check_cuda(ctx, cudaGetLastError(), "k_acc_merge");
}

int bioem_group_logsumexp(bioem_ctx* ctx, const double* d_values, long long n_groups, int group_len, double* d_out) {
    if (!ctx || n_groups < 0 || group_len < 1 || (n_groups > 0 && (!d_values || !d_out))) return BIOEM_ERR_INVALID_ARG;
    if (n_groups == 0) return BIOEM_OK;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "cudaSetDevice");
    // few groups: small blocks, over every SM's float64 pipe (us with 64 and 256 threads: 14,000 groups of 16: 19 and
    // 29; 200,000: 128 and 140); more than 4096 of them: large ones (1e6: 584 and 574; 5e6: 2910 and 2806)
    const int threads = n_groups <= 262144 ? 64 : 256;
    const long long blocks = (n_groups + threads - 1) / threads;
    bioem_launch_begin(ctx, KID_LSE_MERGE);
    k_group_lse<<<(unsigned)(blocks < 4096 ? blocks : 4096), threads, 0, ctx->stream>>>(d_values, n_groups, group_len, d_out);
    bioem_launch_end(ctx, KID_LSE_MERGE);
    return bioem_check_cuda(ctx, cudaGetLastError(), "k_group_lse");
}

__global__ void k_ln1m(const float* __restrict__ x, long long n, float* __restrict__ t) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        t[i] = ln1m(x[i]);
}

int bioem_ln1m(bioem_ctx* ctx, const float* d_x, long long n, float* d_t) {
    if (!ctx || n < 0 || (n > 0 && (!d_x || !d_t))) return BIOEM_ERR_INVALID_ARG;
    if (n == 0) return BIOEM_OK;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "cudaSetDevice");
    const long long blocks = (n + 255) / 256;
    bioem_launch_begin(ctx, KID_LSE_MERGE);
    k_ln1m<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, ctx->stream>>>(d_x, n, d_t);
    bioem_launch_end(ctx, KID_LSE_MERGE);
    return bioem_check_cuda(ctx, cudaGetLastError(), "k_ln1m");
}

int bioem_acc_logP(bioem_ctx* ctx, const double* d_acc, int n_img, double log_norm, double* d_logP) {
    if (!ctx || (n_img > 0 && (!d_acc || !d_logP)) || n_img < 0) return BIOEM_ERR_INVALID_ARG;
    if (n_img == 0) return BIOEM_OK;
    cudaSetDevice(ctx->device);
    bioem_launch_begin(ctx, KID_FINALIZE);
    k_acc_logP<<<(n_img + 255) / 256, 256, 0, ctx->stream>>>(d_acc, n_img, log_norm, d_logP);
    bioem_launch_end(ctx, KID_FINALIZE);
    return bioem_check_cuda(ctx, cudaGetLastError(), "k_acc_logP");
}

}  // extern "C"

// Learned orientation / defocus proposal network: own forward, backward and Adam kernels.
//
// The paper has no learned component; this network proposes where on the orientation x defocus
// grid an image's posterior mass lies, so that only those parameter sets are scored exactly.
//
// Network (input S x S, S = 64 in production: the 128 px image averaged over 2 x 2 pixels and
// standardised per image):
//   conv1 1->C, 3x3, stride 1, pad 1, ReLU       S   x S
//   conv2 C->C, stride 2, ReLU                   S/2
//   conv3 C->C, stride 1, ReLU                   S/2
//   conv4 C->C, stride 2, ReLU                   S/4
//   conv5 C->C, stride 1, ReLU                   S/4
//   conv6 C->C, stride 2, ReLU                   S/8  -> F = C (S/8)^2 features
//   head_q: F -> n_q logits (coarse orientation bins); head_d: F -> n_d logits (defocus bins)
//   loss = mean over the batch of CE(head_q, label_q) + CE(head_d, label_d)
// Parameters are kept in float32 (Adam state and master copy); the forward and backward passes
// read a float16 copy of the weights (rounded after every update).  Activations are float32, NCHW.
// Flat parameter order: for each conv layer W[co][ci][3][3] then b[co]; then Wq[n_q][F], bq[n_q],
// Wd[n_d][F], bd[n_d].
#include <cuda_fp16.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <new>
#include <vector>

#include "bioem_internal.cuh"

namespace {

constexpr int kLayers = 6;
constexpr int kT = 256;
constexpr int kFeatSplits = 16;   // most k splits of the feature gradient (its parts need F kFeatSplits <= C S^2 = 64 F)

struct Layer {
    int cin, cout, stride, hin, hout;
    size_t w_off, b_off;     // offsets in the flat parameter vector
    size_t in_off, out_off;  // activation offsets (per-sample element counts are cin*hin^2, cout*hout^2)
};

// ------------------------------------------------------------------ input preparation
// out[b][y][x] = standardised down x down average of img[b]; per image: zero mean, unit variance over S^2
// (float64 sums per thread, then over lanes and warps in order).  Bound by float64 arithmetic, so few threads
// with many pixels each: a sum over more lanes costs more float64 additions than the pixels.
__global__ void __launch_bounds__(kT) k_downsample_norm(const float* __restrict__ img, int n_in, int down,
                                                        float* __restrict__ out) {
    const int b = blockIdx.x;
    const int S = n_in / down;
    const float* src = img + (size_t)b * n_in * n_in;
    float* dst = out + (size_t)b * S * S;
    __shared__ double r1[kT / 32], r2[kT / 32];
    double s1 = 0.0, s2 = 0.0;
#pragma unroll 4
    for (int i = threadIdx.x; i < S * S; i += kT) {
        const int y = i / S, x = i - y * S;
        float v = 0.f;
        if (down == 2) {
            const float* p = src + (size_t)(2 * y) * n_in + 2 * x;
            v = v + __ldg(p) + __ldg(p + 1) + __ldg(p + n_in) + __ldg(p + n_in + 1);
        } else {
            for (int dy = 0; dy < down; ++dy)
                for (int dx = 0; dx < down; ++dx) v += src[(size_t)(y * down + dy) * n_in + x * down + dx];
        }
        v *= 1.0f / (float)(down * down);
        dst[i] = v;
        const double d = v;
        s1 += d;
        s2 = fma(d, d, s2);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, off);
        s2 += __shfl_xor_sync(0xffffffffu, s2, off);
    }
    if ((threadIdx.x & 31) == 0) {
        r1[threadIdx.x >> 5] = s1;
        r2[threadIdx.x >> 5] = s2;
    }
    __shared__ float stat[2];
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kT / 32; ++w) {
            s1 += r1[w];
            s2 += r2[w];
        }
        const double n = (double)S * S;
        const double mean = s1 / n;
        const double var = s2 / n - mean * mean;
        stat[0] = (float)mean;
        stat[1] = var > 0.0 ? (float)(1.0 / sqrt(var)) : 0.f;
    }
    __syncthreads();
    const float m = stat[0], inv = stat[1];
    for (int i = threadIdx.x; i < S * S; i += kT) dst[i] = (dst[i] - m) * inv;
}

// ------------------------------------------------------------------ convolution
// out[b][co][y][x] = ReLU(b[co] + sum_ci,ky,kx W[co][ci][ky][kx] in[b][ci][y s + ky - 1][x s + kx - 1])
//
// A thread owns XT = 4 neighbouring outputs of one row in CO output channels, so an input row segment
// loaded once serves 3 CO products per value and a weight serves XT; the products of two channels go
// out as one packed FP32 pair.  Every output is still summed in the order (ci, ky, kx) starting from
// the bias, with the taps outside the image left out, so the activations do not depend on the tiling.
// Bound by the FP32 pipe (42 of 73 TFLOP/s at 32 x 32 px, 256 samples: 12-16 warps per SM).  CO = 16 has the
// fewest loads per product; fewer channels per thread are taken where that would leave too few
// blocks (conv_co).  Loading the next channel's rows ahead gained nothing (registers for warps).  VEC: rows read as float4 with the edge
// values from the neighbouring lanes (needs output rows of whole groups of four).
constexpr int XT = 4;
constexpr int kConvT = 128;

// BWD (stride 1): the gradient of the layer's input, din[b][ci][y][x] = sum_co,ky,kx gout[b][co][y + 1 - ky]
// [x + 1 - kx] W[co][ci][ky][kx], the same sum with the channels' roles exchanged and the taps reversed
// (cin, cout are then the layer's output and input channels); no bias, and the ReLU that produced the
// layer's input (mask = that input) is applied to the result instead of in a pass of its own.
template <int CO, int STRIDE, bool VEC, bool BWD>
__global__ void __launch_bounds__(kConvT, 4) k_conv(const float* __restrict__ in, const __half* __restrict__ W,
                                                 const __half* __restrict__ bias, const float* __restrict__ mask,
                                                 int cin, int cout, int hin, int hout, int groups, long long n_tasks,
                                                 float* __restrict__ out) {
    static_assert(!BWD || STRIDE == 1, "the stride-2 input gradient is k_conv_bwd_data2");
    constexpr int NIN = (XT - 1) * STRIDE + 3;   // input columns x0 s - 1 .. x0 s + (XT - 1) s + 1
    extern __shared__ __align__(16) float wsm[];   // [cin * 9][CO], this block's output channels
    const int co0 = blockIdx.y * CO;
    for (int i = threadIdx.x; i < cin * 9 * CO; i += kConvT) {
        const int c = i / (cin * 9), t = i - c * (cin * 9);
        const int ci = t / 9, tap = t - ci * 9;
        const size_t at = BWD ? ((size_t)ci * cout + co0 + c) * 9 + 8 - tap : (size_t)(co0 + c) * cin * 9 + t;
        wsm[t * CO + c] = co0 + c < cout ? __half2float(W[at]) : 0.f;
    }
    __syncthreads();
    const long long task = (long long)blockIdx.x * kConvT + threadIdx.x;
    const bool live = task < n_tasks;
    const long long tk = live ? task : n_tasks - 1;
    const long long row_id = tk / groups;
    const int xg = (int)(tk - row_id * groups);
    const int b = (int)(row_id / hout);
    const int y = (int)(row_id - (long long)b * hout);
    const int x0 = xg * XT;
    const int lane = threadIdx.x & 31;
    float2 acc[XT][CO / 2];
#pragma unroll
    for (int p = 0; p < CO / 2; ++p) {
        const int c = co0 + 2 * p;
        const float2 bv = make_float2(!BWD && c < cout ? __half2float(bias[c]) : 0.f,
                                      !BWD && c + 1 < cout ? __half2float(bias[c + 1]) : 0.f);
#pragma unroll
        for (int i = 0; i < XT; ++i) acc[i][p] = bv;
    }
    const float* ic = in + (size_t)b * cin * hin * hin;
#pragma unroll 1
    for (int ci = 0; ci < cin; ++ci, ic += hin * hin) {
        float v[3][NIN];
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
            const int iy = y * STRIDE + ky - 1;
            const float* row = ic + min(max(iy, 0), hin - 1) * hin;   // clamped: an outside row is not used
            if constexpr (VEC) {
#pragma unroll
                for (int k = 0; k < STRIDE; ++k) {
                    const float4 q = __ldg(reinterpret_cast<const float4*>(row + x0 * STRIDE) + k);
                    v[ky][1 + 4 * k] = q.x; v[ky][2 + 4 * k] = q.y; v[ky][3 + 4 * k] = q.z; v[ky][4 + 4 * k] = q.w;
                }
                v[ky][0] = __shfl_up_sync(0xffffffffu, v[ky][4 * STRIDE], 1);
                if (lane == 0 && xg > 0) v[ky][0] = __ldg(row + x0 * STRIDE - 1);
                if constexpr (STRIDE == 1) {
                    v[ky][NIN - 1] = __shfl_down_sync(0xffffffffu, v[ky][1], 1);
                    if (lane == 31 && x0 + XT < hin) v[ky][NIN - 1] = __ldg(row + x0 + XT);
                }
            } else {
#pragma unroll
                for (int k = 0; k < NIN; ++k) {
                    const int ix = x0 * STRIDE + k - 1;
                    v[ky][k] = (ix >= 0 && ix < hin) ? __ldg(row + ix) : 0.f;
                }
            }
        }
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
            const int iy = y * STRIDE + ky - 1;
            if (iy < 0 || iy >= hin) continue;
            const float4* wp = reinterpret_cast<const float4*>(wsm + (size_t)(ci * 9 + ky * 3) * CO);
#pragma unroll
            for (int kx = 0; kx < 3; ++kx)
#pragma unroll
                for (int p = 0; p < CO / 4; ++p) {
                    const float4 w = wp[kx * (CO / 4) + p];
#pragma unroll
                    for (int i = 0; i < XT; ++i) {
                        const int ix = (x0 + i) * STRIDE + kx - 1;
                        // only the first and (stride 1) the last column of a row can fall outside
                        if (VEC && !(i * STRIDE + kx == 0) && !(STRIDE == 1 && i + kx == XT + 1)) {
                        } else if (ix < 0 || ix >= hin) {
                            continue;
                        }
                        const float x = v[ky][i * STRIDE + kx];
                        acc[i][2 * p] = __ffma2_rn(make_float2(x, x), make_float2(w.x, w.y), acc[i][2 * p]);
                        acc[i][2 * p + 1] = __ffma2_rn(make_float2(x, x), make_float2(w.z, w.w), acc[i][2 * p + 1]);
                    }
                }
        }
    }
    if (!live) return;
#pragma unroll
    for (int c = 0; c < CO; ++c) {
        if (co0 + c >= cout) break;
        const size_t at = (((size_t)b * cout + co0 + c) * hout + y) * hout + x0;
        float* o = out + at;
        float r[XT];
#pragma unroll
        for (int i = 0; i < XT; ++i) {
            const float a = (c & 1) ? acc[i][c / 2].y : acc[i][c / 2].x;
            if constexpr (BWD) r[i] = (VEC || x0 + i < hout) && mask[at + i] > 0.f ? a : 0.f;
            else r[i] = a > 0.f ? a : 0.f;
        }
        if constexpr (VEC) {
            *reinterpret_cast<float4*>(o) = make_float4(r[0], r[1], r[2], r[3]);
        } else {
#pragma unroll
            for (int i = 0; i < XT; ++i)
                if (x0 + i < hout) o[i] = r[i];
        }
    }
}

// The input gradient of a stride-2 layer, masked by the ReLU that produced that input:
//   din[b][ci][iy][ix] = sum over (co, ky, kx) with iy = 2 y + ky - 1, ix = 2 x + kx - 1 of gout[b][co][y][x] W[co][ci][ky][kx].
// Every 2 x 2 block of the input takes 9 taps (1 + 2 + 2 + 4) from the outputs at (y, y + 1) x (x, x + 1), so a
// thread owns the blocks of four neighbouring output columns x0 .. x0 + 3 in two input channels pairs
// (CI = 4) and forms no product that falls on a hole of the stride.
constexpr int CI2 = 4;
template <bool VEC>
__global__ void __launch_bounds__(kConvT) k_conv_bwd_data2(const float* __restrict__ gout, const __half* __restrict__ W,
                                                           const float* __restrict__ mask, int cin, int cout, int hin,
                                                           int hout, int groups, long long n_tasks,
                                                           float* __restrict__ din) {
    extern __shared__ __align__(16) float wsm[];   // [cout * 9][CI2], this block's input channels
    const int ci0 = blockIdx.y * CI2;
    for (int i = threadIdx.x; i < cout * 9 * CI2; i += kConvT) {
        const int c = i % CI2, t = i / CI2;
        const int co = t / 9, tap = t - co * 9;
        wsm[i] = ci0 + c < cin ? __half2float(W[((size_t)co * cin + ci0 + c) * 9 + tap]) : 0.f;
    }
    __syncthreads();
    const long long task = (long long)blockIdx.x * kConvT + threadIdx.x;
    const bool live = task < n_tasks;
    const long long tk = live ? task : n_tasks - 1;
    const long long row_id = tk / groups;
    const int xg = (int)(tk - row_id * groups);
    const int b = (int)(row_id / hout);
    const int y = (int)(row_id - (long long)b * hout);
    const int x0 = xg * XT;
    const int lane = threadIdx.x & 31;
    float2 acc[2][2 * XT][CI2 / 2];   // [input row 2y, 2y + 1][input column 2 x0 + .][channel pair]
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int i = 0; i < 2 * XT; ++i)
#pragma unroll
            for (int p = 0; p < CI2 / 2; ++p) acc[r][i][p] = make_float2(0.f, 0.f);
    const float* gc = gout + (size_t)b * cout * hout * hout;
    const bool below = y + 1 < hout;
#pragma unroll 1
    for (int co = 0; co < cout; ++co, gc += hout * hout) {
        float g[2][XT + 1];   // rows y, y + 1; columns x0 .. x0 + 4; 0 outside
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float* row = gc + (size_t)min(y + r, hout - 1) * hout;
            if constexpr (VEC) {
                const float4 q = __ldg(reinterpret_cast<const float4*>(row + x0));
                g[r][0] = q.x; g[r][1] = q.y; g[r][2] = q.z; g[r][3] = q.w;
                g[r][4] = __shfl_down_sync(0xffffffffu, q.x, 1);
                if (lane == 31 && x0 + XT < hout) g[r][4] = __ldg(row + x0 + XT);
                if (x0 + XT >= hout) g[r][4] = 0.f;
            } else {
#pragma unroll
                for (int i = 0; i <= XT; ++i) g[r][i] = x0 + i < hout ? __ldg(row + x0 + i) : 0.f;
            }
            if (r == 1 && !below)
#pragma unroll
                for (int i = 0; i <= XT; ++i) g[r][i] = 0.f;
        }
        const float4* wp = reinterpret_cast<const float4*>(wsm + (size_t)co * 9 * CI2);
        // input row 2y takes ky = 1 of row y; row 2y + 1 takes ky = 2 of row y and ky = 0 of row y + 1;
        // columns alike
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
            const int r_in = ky == 1 ? 0 : 1, r_g = ky == 0 ? 1 : 0;
#pragma unroll
            for (int kx = 0; kx < 3; ++kx) {
                const int c_in = kx == 1 ? 0 : 1, c_g = kx == 0 ? 1 : 0;
                const float4 w = wp[ky * 3 + kx];
#pragma unroll
                for (int i = 0; i < XT; ++i) {
                    const float2 v = make_float2(g[r_g][i + c_g], g[r_g][i + c_g]);
                    acc[r_in][2 * i + c_in][0] = __ffma2_rn(v, make_float2(w.x, w.y), acc[r_in][2 * i + c_in][0]);
                    acc[r_in][2 * i + c_in][1] = __ffma2_rn(v, make_float2(w.z, w.w), acc[r_in][2 * i + c_in][1]);
                }
            }
        }
    }
    if (!live) return;
#pragma unroll
    for (int c = 0; c < CI2; ++c) {
        if (ci0 + c >= cin) break;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const size_t at = (((size_t)b * cin + ci0 + c) * hin + 2 * y + r) * hin + 2 * x0;
            float v[2 * XT];
#pragma unroll
            for (int i = 0; i < 2 * XT; ++i) v[i] = (c & 1) ? acc[r][i][c / 2].y : acc[r][i][c / 2].x;
            if constexpr (VEC) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const float4 m = *reinterpret_cast<const float4*>(mask + at + 4 * k);
                    *reinterpret_cast<float4*>(din + at + 4 * k) =
                        make_float4(m.x > 0.f ? v[4 * k] : 0.f, m.y > 0.f ? v[4 * k + 1] : 0.f,
                                    m.z > 0.f ? v[4 * k + 2] : 0.f, m.w > 0.f ? v[4 * k + 3] : 0.f);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 2 * XT; ++i)
                    if (2 * x0 + i < hin) din[at + i] = mask[at + i] > 0.f ? v[i] : 0.f;
            }
        }
    }
}

// Weight gradients gW[co][ci][ky][kx] = sum_{b,y,x} gout[b][co][y][x] in[b][ci][y s + ky - 1][x s + kx - 1] and bias
// gradients gb[co] = sum_{b,y,x} gout[b][co][y][x], as partial sums per block (k_conv_wgrad_sum adds them in
// block order: deterministic).  A block holds 32 x 32 channels x 9 taps, 2 x 2 x 9 sums per thread, and
// walks over tiles of WR output rows x GW columns of one sample staged in shared memory (outside values
// zero), four columns at a time: 144 products per 14-16 shared reads, against one read per product when
// each (co, ci) pair was a block of its own.  Bound by the FP32 pipe.  All of a tile's loads are in flight
// together (row by row, each waited for, they took longer than the products: 281 us for the 32 x 32 px stride-1
// layer of 256 samples against 115).  Channel strides are 4 x odd floats, so the 16-byte reads of 8
// neighbouring channels do not conflict.
// Only products of a gradient that is not 0 with a value inside the image count: a value that is not finite
// behind a ReLU that stopped it (an image of NaN gives an input of NaN, and first activations of 0) must not
// reach the sums.  The fast path forms 0 x value everywhere, the same sum while all values are finite; a tile
// that holds another value takes the slow one.
constexpr int kWgT = 256, kWgC = 32, kWgX = 64;

__host__ __device__ constexpr int odd4(int n) { return ((n + 3) / 4 | 1) * 4; }   // >= n, 4 x odd

template <int STRIDE, int GW>
struct WgTile {
    static constexpr int WR = STRIDE == 1 ? (GW == 8 ? 8 : 128 / GW) : 64 / GW;   // output rows
    static constexpr int IR = (WR - 1) * STRIDE + 3;                                // input rows
    static constexpr int IW = STRIDE == 1 ? GW + 8 : 2 * GW + 4;   // staged input row: column ix at ix + 4
    static constexpr int GCH = odd4(WR * GW), ICH = odd4(IR * IW);   // channel strides
    static constexpr size_t SMEM = (size_t)kWgC * (GCH + ICH) * sizeof(float);
};

// chk + 0 v: NaN if chk or a value of v is not finite, else chk
__device__ __forceinline__ float not_finite(float4 v, float chk) {
    return fmaf(v.w, 0.f, fmaf(v.z, 0.f, fmaf(v.y, 0.f, fmaf(v.x, 0.f, chk))));
}

// VEC: rows of whole groups of four (16-byte loads).
template <int STRIDE, int GW, bool VEC>
__global__ void __launch_bounds__(kWgT, 2) k_conv_wgrad(const float* __restrict__ gout, const float* __restrict__ in,
                                                        int B, int cin, int cout, int hin, int hout,
                                                        float* __restrict__ part) {
    using W = WgTile<STRIDE, GW>;
    constexpr int WR = W::WR, IR = W::IR, IW = W::IW, GCH = W::GCH, ICH = W::ICH;
    extern __shared__ __align__(16) float sm[];
    float* gs = sm;                   // [32 co][WR][GW]
    float* is = sm + kWgC * GCH;      // [32 ci][IR][IW]
    const int nci = (cin + kWgC - 1) / kWgC;
    const int co0 = (int)blockIdx.y / nci * kWgC, ci0 = (int)blockIdx.y % nci * kWgC;
    const int tc = threadIdx.x & 15, to = threadIdx.x >> 4;   // ci = ci0 + tc + 16 j, co = co0 + to + 16 i
    float acc[2][2][9], sb[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int k = 0; k < 9; ++k) acc[i][j][k] = 0.f;
    // four values of a row from column x (all of them inside or outside the row with VEC)
    auto load4 = [](const float* row, int x, int n, bool ok) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (VEC) {
            if (ok && x < n) v = __ldg(reinterpret_cast<const float4*>(row + x));
        } else if (ok) {
            if (x < n) v.x = __ldg(row + x);
            if (x + 1 < n) v.y = __ldg(row + x + 1);
            if (x + 2 < n) v.z = __ldg(row + x + 2);
            if (x + 3 < n) v.w = __ldg(row + x + 3);
        }
        return v;
    };
    const int tiles_x = (hout + GW - 1) / GW, tiles = (hout + WR - 1) / WR * tiles_x;
    const long long units = (long long)B * tiles;
    for (long long u = blockIdx.x; u < units; u += gridDim.x) {
        const int b = (int)(u / tiles), t = (int)(u - (long long)b * tiles);
        const int y0 = t / tiles_x * WR, xs = t % tiles_x * GW;
        constexpr int NG = kWgC * WR * (GW / 4), NI = kWgC * IR * (GW * STRIDE / 4), NE = kWgC * IR * 2;
        constexpr int PG = (NG + kWgT - 1) / kWgT, PI = (NI + kWgT - 1) / kWgT, PE = (NE + kWgT - 1) / kWgT;
        float4 vg[PG], vi[PI];
        float ve[PE];
#pragma unroll
        for (int k = 0; k < PG; ++k) {
            const int e = threadIdx.x + k * kWgT, x = e % (GW / 4) * 4, y = e / (GW / 4) % WR, c = e / (GW / 4 * WR);
            const bool ok = e < NG && co0 + c < cout && y0 + y < hout;
            vg[k] = load4(gout + (((size_t)b * cout + co0 + c) * hout + y0 + y) * hout, xs + x, hout, ok);
        }
#pragma unroll
        for (int k = 0; k < PI; ++k) {
            constexpr int Q = GW * STRIDE / 4;
            const int e = threadIdx.x + k * kWgT, x = e % Q * 4, y = e / Q % IR, c = e / (Q * IR);
            const int iy = y0 * STRIDE + y - 1;
            const bool ok = e < NI && ci0 + c < cin && iy >= 0 && iy < hin;
            vi[k] = load4(in + (((size_t)b * cin + ci0 + c) * hin + iy) * hin, xs * STRIDE + x, hin, ok);
        }
#pragma unroll
        for (int k = 0; k < PE; ++k) {   // the columns left and right of the tile
            const int e = threadIdx.x + k * kWgT, y = e / 2 % IR, c = e / (2 * IR);
            const int iy = y0 * STRIDE + y - 1, ix = e & 1 ? (xs + GW) * STRIDE : xs * STRIDE - 1;
            const bool ok = e < NE && ci0 + c < cin && iy >= 0 && iy < hin && ix >= 0 && ix < hin;
            ve[k] = ok ? __ldg(in + (((size_t)b * cin + ci0 + c) * hin + iy) * hin + ix) : 0.f;
        }
        __syncthreads();   // the previous tile has been read
        float chk = 0.f;   // NaN once a staged value is not finite
#pragma unroll
        for (int k = 0; k < PG; ++k) {
            const int e = threadIdx.x + k * kWgT, x = e % (GW / 4) * 4, y = e / (GW / 4) % WR, c = e / (GW / 4 * WR);
            if (e < NG) *reinterpret_cast<float4*>(gs + c * GCH + y * GW + x) = vg[k];
            chk = not_finite(vg[k], chk);
        }
#pragma unroll
        for (int k = 0; k < PI; ++k) {
            constexpr int Q = GW * STRIDE / 4;
            const int e = threadIdx.x + k * kWgT, x = e % Q * 4, y = e / Q % IR, c = e / (Q * IR);
            if (e < NI) *reinterpret_cast<float4*>(is + c * ICH + y * IW + 4 + x) = vi[k];
            chk = not_finite(vi[k], chk);
        }
#pragma unroll
        for (int k = 0; k < PE; ++k) {
            const int e = threadIdx.x + k * kWgT, y = e / 2 % IR, c = e / (2 * IR);
            if (e < NE && !(STRIDE == 2 && (e & 1))) is[c * ICH + y * IW + (e & 1 ? 4 + GW * STRIDE : 3)] = ve[k];
            chk = fmaf(ve[k], 0.f, chk);
        }
        if (__syncthreads_or(!(chk == 0.f))) {
#pragma unroll 1
            for (int q = 0; q < WR * GW; ++q) {
                const int y = q / GW, x = q - y * GW;
                const float g[2] = {gs[to * GCH + q], gs[(to + 16) * GCH + q]};
                sb[0] += g[0];
                sb[1] += g[1];
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) {
                    const int iy = (y0 + y) * STRIDE + ky - 1;
                    if (iy < 0 || iy >= hin) continue;
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) {
                        const int ix = (xs + x) * STRIDE + kx - 1;
                        if (ix < 0 || ix >= hin) continue;
                        const int at = (y * STRIDE + ky) * IW + x * STRIDE + kx + 3;
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const float v = is[(tc + 16 * j) * ICH + at];
#pragma unroll
                            for (int i = 0; i < 2; ++i)
                                if (g[i] != 0.f) acc[i][j][ky * 3 + kx] = fmaf(g[i], v, acc[i][j][ky * 3 + kx]);
                        }
                    }
                }
            }
            continue;
        }
#pragma unroll 1
        for (int y = 0; y < WR; ++y) {
            const float* gp = gs + to * GCH + y * GW;
            const float* ip = is + tc * ICH + y * STRIDE * IW + 4;
            float left[2][3];   // the value before the next group of columns
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) left[j][ky] = ip[16 * j * ICH + ky * IW - 1];
#pragma unroll 2
            for (int x0 = 0; x0 < GW; x0 += 4) {
                float g[2][4];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float4 v = *reinterpret_cast<const float4*>(gp + 16 * i * GCH + x0);
                    g[i][0] = v.x; g[i][1] = v.y; g[i][2] = v.z; g[i][3] = v.w;
                    sb[i] += (v.x + v.y) + (v.z + v.w);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky) {
                        const float* row = ip + 16 * j * ICH + ky * IW + x0 * STRIDE;
                        float v[4 * STRIDE + 2];
                        v[0] = left[j][ky];
#pragma unroll
                        for (int q = 0; q < STRIDE; ++q) {
                            const float4 w = *reinterpret_cast<const float4*>(row + 4 * q);
                            v[4 * q + 1] = w.x; v[4 * q + 2] = w.y; v[4 * q + 3] = w.z; v[4 * q + 4] = w.w;
                        }
                        left[j][ky] = v[4 * STRIDE];
                        v[4 * STRIDE + 1] = STRIDE == 1 ? row[4] : 0.f;   // stride 2 ends inside the group
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int kx = 0; kx < 3; ++kx)
#pragma unroll
                                for (int x = 0; x < 4; ++x)
                                    acc[i][j][ky * 3 + kx] = fmaf(g[i][x], v[x * STRIDE + kx], acc[i][j][ky * 3 + kx]);
                    }
            }
        }
    }
    float* o = part + (size_t)blockIdx.x * ((size_t)cout * cin * 9 + cout);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int co = co0 + to + 16 * i;
        if (co >= cout) continue;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int ci = ci0 + tc + 16 * j;
            if (ci >= cin) continue;
#pragma unroll
            for (int k = 0; k < 9; ++k) o[((size_t)co * cin + ci) * 9 + k] = acc[i][j][k];
        }
        if (ci0 == 0 && tc == 0) o[(size_t)cout * cin * 9 + co] = sb[i];
    }
}

// The same for the first layer (one input channel, stride 1): two output channels per warp, 16 per block, its
// lanes over groups of four columns of a tile of 16 rows.  Bound by reading gout once.  Which products count: as
// above, the slow path for a group of columns whose gradients or a tile whose inputs are not all finite.
constexpr int kW1Rows = 16, kW1C = 16;
__global__ void __launch_bounds__(kWgT) k_conv_wgrad1(const float* __restrict__ gout, const float* __restrict__ in,
                                                      int B, int cout, int h, float* __restrict__ part) {
    extern __shared__ __align__(16) float is[];   // [kW1Rows + 2][iw], column ix + 1
    const int gw = h < kWgX ? (h + 3) / 4 * 4 : kWgX, iw = gw + 4, q4 = gw / 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int CW = kW1C / (kWgT / 32);   // output channels per warp
    float acc[CW][10];
#pragma unroll
    for (int c = 0; c < CW; ++c)
#pragma unroll
        for (int k = 0; k < 10; ++k) acc[c][k] = 0.f;
    const int tiles_x = (h + gw - 1) / gw, tiles = (h + kW1Rows - 1) / kW1Rows * tiles_x;
    const long long units = (long long)B * tiles;
    const bool vec = h % 4 == 0;
    const int cw = blockIdx.y * kW1C + warp * CW;
    for (long long u = blockIdx.x; u < units; u += gridDim.x) {
        const int b = (int)(u / tiles), t = (int)(u - (long long)b * tiles);
        const int y0 = t / tiles_x * kW1Rows, xs = t % tiles_x * gw;
        __syncthreads();
        float chk = 0.f;   // NaN once an input is not finite
        for (int i = threadIdx.x; i < (kW1Rows + 2) * iw; i += kWgT) {
            const int y = i / iw, x = i - y * iw;
            const int iy = y0 + y - 1, ix = xs + x - 1;
            const float v = iy >= 0 && iy < h && ix >= 0 && ix < h ? __ldg(in + ((size_t)b * h + iy) * h + ix) : 0.f;
            is[i] = v;
            chk = fmaf(v, 0.f, chk);
        }
        const bool odd = __syncthreads_or(!(chk == 0.f));
        const int rows = min(kW1Rows, h - y0);
#pragma unroll 2
        for (int e = lane; e < rows * q4; e += 32) {
            const int y = e / q4, x0 = (e - y * q4) * 4;
            if (xs + x0 >= h) continue;
            float g[CW][4];
#pragma unroll
            for (int c = 0; c < CW; ++c) {
                const float* gp = gout + (((size_t)b * cout + min(cw + c, cout - 1)) * h + y0 + y) * h + xs + x0;
                if (vec) {
                    const float4 v = __ldg(reinterpret_cast<const float4*>(gp));
                    g[c][0] = v.x; g[c][1] = v.y; g[c][2] = v.z; g[c][3] = v.w;
                } else {
#pragma unroll
                    for (int x = 0; x < 4; ++x) g[c][x] = xs + x0 + x < h ? __ldg(gp + x) : 0.f;
                }
            }
            float v[3][6];
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
                const float* row = is + (y + ky) * iw + x0;
                const float4 w = *reinterpret_cast<const float4*>(row);
                const float2 w2 = *reinterpret_cast<const float2*>(row + 4);
                v[ky][0] = w.x; v[ky][1] = w.y; v[ky][2] = w.z; v[ky][3] = w.w; v[ky][4] = w2.x; v[ky][5] = w2.y;
            }
            float gchk = 0.f;
#pragma unroll
            for (int c = 0; c < CW; ++c) gchk = not_finite(make_float4(g[c][0], g[c][1], g[c][2], g[c][3]), gchk);
            if (odd || !(gchk == 0.f)) {
#pragma unroll
                for (int c = 0; c < CW; ++c)
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
#pragma unroll
                        for (int k = 0; k < 9; ++k) {
                            const int iy = y0 + y + k / 3 - 1, ix = xs + x0 + x + k % 3 - 1;
                            if (g[c][x] != 0.f && iy >= 0 && iy < h && ix >= 0 && ix < h)
                                acc[c][k] = fmaf(g[c][x], v[k / 3][x + k % 3], acc[c][k]);
                        }
                        acc[c][9] += g[c][x];
                    }
                continue;
            }
#pragma unroll
            for (int c = 0; c < CW; ++c)
#pragma unroll
                for (int x = 0; x < 4; ++x) {
#pragma unroll
                    for (int k = 0; k < 9; ++k) acc[c][k] = fmaf(g[c][x], v[k / 3][x + k % 3], acc[c][k]);
                    acc[c][9] += g[c][x];
                }
        }
    }
    float* o = part + (size_t)blockIdx.x * ((size_t)cout * 9 + cout);
#pragma unroll
    for (int c = 0; c < CW; ++c) {
        const int co = cw + c;
#pragma unroll
        for (int k = 0; k < 10; ++k) {
            float s = acc[c][k];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (lane == 0 && co < cout) o[k < 9 ? (size_t)co * 9 + k : (size_t)cout * 9 + co] = s;
        }
    }
}

// out[i] = sum over blocks of part[block][i], 8 runs of blocks in order, then the runs; the first n_w
// values are the weights' gradients, the rest the biases'.
__global__ void __launch_bounds__(kT) k_conv_wgrad_sum(const float* __restrict__ part, int blocks, int n_w, int n,
                                                       float* __restrict__ gW, float* __restrict__ gb) {
    __shared__ float red[8][32];
    const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + c;
    float s = 0.f;
    if (i < n)
        for (int k = g; k < blocks; k += 8) s += part[(size_t)k * n + i];
    red[g][c] = s;
    __syncthreads();
    if (g == 0 && i < n) {
        for (int k = 1; k < 8; ++k) s += red[k][c];
        if (i < n_w) gW[i] = s;
        else gb[i - n_w] = s;
    }
}

// ------------------------------------------------------------------ dense layers (tiled GEMM)
// C(m, n) = sum_k A(m, k) B(n, k), k ascending in one FP32 accumulator per output.  128 threads, a
// TM x TN tile, MT x NT outputs per thread (rows in packed FP32 pairs), KT of k per step in two shared
// buffers, the next step's operands held in registers meanwhile.  Bound by the FP32 pipe; each thread's
// share of an operand lies on a few rows whose addresses are formed once (per element they
// took half as many instructions as the products) and whose values stay as loaded until they are stored
// (converting float16 weights at the load waited for it): 163 -> 128 us for the logits of 256 samples, 353 -> 110
// for their feature gradients.
// The two heads form one product (their columns or rows follow one another).
constexpr int kGemmT = 128, KT = 32;

// One operand of a tile: ROWS rows (m or n), KT of k.  ADJ: consecutive k are adjacent in memory; a warp then
// takes 8 k x 4 rows per load (full 32-byte sectors, conflict-free transposed stores), else a run of rows.
template <int ROWS, bool ADJ, class T>
struct Operand {
    static constexpr int PER = ROWS * KT / kGemmT, NP = ADJ ? ROWS / 16 : 1;
    const T* p[NP];
    bool ok[NP];
    long long ld;   // step of k when not ADJ
    T v[PER];       // as loaded: converting here would wait for the load
    static __device__ __forceinline__ int row(int i) {
        return ADJ ? ((int)threadIdx.x >> 3) + 16 * (i % NP) : (int)threadIdx.x % ROWS;
    }
    static __device__ __forceinline__ int k(int i) {
        return ADJ ? ((int)threadIdx.x & 7) + 8 * (i / NP) : (int)threadIdx.x / ROWS + i * (kGemmT / ROWS);
    }
    __device__ __forceinline__ void fetch(int k0, int ke) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int kk = k0 + k(i);
            v[i] = ok[i % NP] && kk < ke ? p[i % NP][ADJ ? (long long)kk : kk * ld] : T(0.f);
        }
    }
    template <int LD>
    __device__ __forceinline__ void stage(float (&S)[KT][LD]) const {
#pragma unroll
        for (int i = 0; i < PER; ++i) S[k(i)][row(i)] = (float)v[i];
    }
};

template <int TM, int TN, int MT, int NT, class OP>
__global__ void __launch_bounds__(kGemmT) k_gemm(const OP op, int k_per_split, int K) {
    static_assert(TM / MT * (TN / NT) == kGemmT && MT % 4 == 0 && NT % 4 == 0, "one MT x NT block per thread");
    __shared__ __align__(16) float As[2][KT][TM + 4], Bs[2][KT][TN + 4];
    const int tn = threadIdx.x % (TN / NT), tm = threadIdx.x / (TN / NT);
    const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
    const int kb = blockIdx.z * k_per_split, ke = min(K, kb + k_per_split);
    float2 acc[MT / 2][NT];
#pragma unroll
    for (int i = 0; i < MT / 2; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j) acc[i][j] = make_float2(0.f, 0.f);
    Operand<TM, OP::AK, typename OP::TA> A;
    Operand<TN, OP::BK, typename OP::TB> B;
#pragma unroll
    for (int i = 0; i < A.NP; ++i) A.ok[i] = op.a(m0 + A.row(i), A.p[i], A.ld);
#pragma unroll
    for (int i = 0; i < B.NP; ++i) B.ok[i] = op.b(n0 + B.row(i), B.p[i], B.ld);
    A.fetch(kb, ke);
    B.fetch(kb, ke);
    A.stage(As[0]);
    B.stage(Bs[0]);
    __syncthreads();
    int buf = 0;
    for (int k0 = kb; k0 < ke; k0 += KT, buf ^= 1) {
        const bool more = k0 + KT < ke;
        if (more) {
            A.fetch(k0 + KT, ke);
            B.fetch(k0 + KT, ke);
        }
#pragma unroll
        for (int kk = 0; kk < KT; ++kk) {
            float2 a[MT / 2];
            float bv[NT];
#pragma unroll
            for (int q = 0; q < MT / 4; ++q) {
                const float4 t = *reinterpret_cast<const float4*>(&As[buf][kk][tm * MT + 4 * q]);
                a[2 * q] = make_float2(t.x, t.y);
                a[2 * q + 1] = make_float2(t.z, t.w);
            }
            // a thread's columns in groups of four TN / (NT / 4) apart: conflict-free 16-byte reads
#pragma unroll
            for (int q = 0; q < NT / 4; ++q) {
                const float4 t = *reinterpret_cast<const float4*>(&Bs[buf][kk][q * (4 * TN / NT) + tn * 4]);
                bv[4 * q] = t.x; bv[4 * q + 1] = t.y; bv[4 * q + 2] = t.z; bv[4 * q + 3] = t.w;
            }
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int i = 0; i < MT / 2; ++i) acc[i][j] = __ffma2_rn(a[i], make_float2(bv[j], bv[j]), acc[i][j]);
        }
        if (more) {
            A.stage(As[buf ^ 1]);
            B.stage(Bs[buf ^ 1]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
            op.store(m0 + tm * MT + i, n0 + (j / 4) * (4 * TN / NT) + tn * 4 + (j & 3), (int)blockIdx.z,
                     (i & 1) ? acc[i / 2][j].y : acc[i / 2][j].x);
}

// The products.  op.a(m, p, ld) / op.b(n, p, ld): the row's address at k = 0 and (not ADJ) the step of k; false
// outside the product.

// Both heads' logits: m = sample, n = orientation bins then defocus bins, k = feature.
struct HeadFwd {
    static constexpr bool AK = true, BK = true;
    using TA = float;
    using TB = __half;
    const float* feat;
    const __half *wq, *bq, *wd, *bd;
    float *lq, *ld;
    int B, nq, nd, F;
    __device__ __forceinline__ bool a(int m, const float*& p, long long&) const {
        p = feat + (size_t)min(m, B - 1) * F;
        return m < B;
    }
    __device__ __forceinline__ bool b(int n, const __half*& p, long long&) const {
        p = n < nq ? wq + (size_t)n * F : wd + (size_t)min(n - nq, nd - 1) * F;
        return n < nq + nd;
    }
    __device__ __forceinline__ void store(int m, int n, int, float v) const {
        if (m >= B || n >= nq + nd) return;
        if (n < nq) lq[(size_t)m * nq + n] = v + __half2float(bq[n]);
        else ld[(size_t)m * nd + n - nq] = v + __half2float(bd[n - nq]);
    }
};

// Both heads' weight gradients: m = bin, n = feature, k = sample.
struct HeadGradW {
    static constexpr bool AK = false, BK = false;
    using TA = float;
    using TB = float;
    const float *glq, *gld, *feat;
    float *gwq, *gwd;
    int B, nq, nd, F;
    __device__ __forceinline__ bool a(int m, const float*& p, long long& ld) const {
        p = m < nq ? glq + m : gld + min(m - nq, nd - 1);
        ld = m < nq ? nq : nd;
        return m < nq + nd;
    }
    __device__ __forceinline__ bool b(int n, const float*& p, long long& ld) const {
        p = feat + min(n, F - 1);
        ld = F;
        return n < F;
    }
    __device__ __forceinline__ void store(int m, int n, int, float v) const {
        if (m >= nq + nd || n >= F) return;
        if (m < nq) gwq[(size_t)m * F + n] = v;
        else gwd[(size_t)(m - nq) * F + n] = v;
    }
};

// Feature gradients from the orientation head, split over k: m = sample, n = feature, k = orientation bin;
// part[split][m][n], summed by k_feat_grad.
struct HeadGradX {
    static constexpr bool AK = true, BK = false;
    using TA = float;
    using TB = __half;
    const float* glq;
    const __half* wq;
    float* part;
    int B, nq, F;
    __device__ __forceinline__ bool a(int m, const float*& p, long long&) const {
        p = glq + (size_t)min(m, B - 1) * nq;
        return m < B;
    }
    __device__ __forceinline__ bool b(int n, const __half*& p, long long& ld) const {
        p = wq + min(n, F - 1);
        ld = F;
        return n < F;
    }
    __device__ __forceinline__ void store(int m, int n, int z, float v) const {
        if (m < B && n < F) part[((size_t)z * B + m) * F + n] = v;
    }
};

// gfeat = the sum of the k splits plus the defocus head's share, back through the ReLU whose output is feat.
__global__ void __launch_bounds__(kT) k_feat_grad(const float* __restrict__ part, int splits, int B, int F,
                                                  const float* __restrict__ gld, const __half* __restrict__ wd, int nd,
                                                  const float* __restrict__ feat, float* __restrict__ gfeat) {
    const size_t n = (size_t)B * F;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int b = (int)(i / F), f = (int)(i - (size_t)b * F);
        float s = 0.f;
        for (int z = 0; z < splits; ++z) s += part[(size_t)z * n + i];
        for (int d = 0; d < nd; ++d) s = fmaf(gld[(size_t)b * nd + d], __half2float(wd[(size_t)d * F + f]), s);
        gfeat[i] = feat[i] > 0.f ? s : 0.f;
    }
}

// Column sums of both heads' logit gradients (the bias gradients), fixed order: 8 row groups per 32
// columns, then the groups.
__global__ void __launch_bounds__(kT) k_colsum(const float* __restrict__ gq, int nq, const float* __restrict__ gd,
                                               int nd, int M, float* __restrict__ outq, float* __restrict__ outd) {
    __shared__ float red[8][32];
    const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int qb = (nq + 31) / 32;
    const bool second = (int)blockIdx.x >= qb;
    const float* G = second ? gd : gq;
    const int N = second ? nd : nq, n = ((int)blockIdx.x - (second ? qb : 0)) * 32 + c;
    float s = 0.f;
    if (n < N)
        for (int m = g; m < M; m += 8) s += G[(size_t)m * N + n];
    red[g][c] = s;
    __syncthreads();
    if (g == 0 && n < N) {
        for (int k = 1; k < 8; ++k) s += red[k][c];
        (second ? outd : outq)[n] = s;
    }
}

// ------------------------------------------------------------------ loss
// Per sample: log-softmax of both heads, loss = -lq[label_q] - ld[label_d]; gradients
// (softmax - onehot) / B written over the logits.  loss_out[b] (may be null).
__global__ void __launch_bounds__(kT) k_softmax_ce(float* __restrict__ lq, int nq, float* __restrict__ ld, int nd,
                                                   const int* __restrict__ yq, const int* __restrict__ yd, int B,
                                                   float* __restrict__ loss_out) {
    const int b = blockIdx.x;
    __shared__ float red[kT];
    __shared__ float stat[2];
    float loss = 0.f;
    for (int head = 0; head < 2; ++head) {
        float* l = head == 0 ? lq + (size_t)b * nq : ld + (size_t)b * nd;
        const int n = head == 0 ? nq : nd;
        const int y = head == 0 ? yq[b] : yd[b];
        float m = -INFINITY;
        for (int i = threadIdx.x; i < n; i += blockDim.x) m = fmaxf(m, l[i]);
        red[threadIdx.x] = m;
        __syncthreads();
        for (int st = blockDim.x / 2; st > 0; st >>= 1) {
            if (threadIdx.x < st) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + st]);
            __syncthreads();
        }
        m = red[0];
        __syncthreads();
        float s = 0.f;
        for (int i = threadIdx.x; i < n; i += blockDim.x) s += expf(l[i] - m);
        red[threadIdx.x] = s;
        __syncthreads();
        for (int st = blockDim.x / 2; st > 0; st >>= 1) {
            if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            stat[0] = m + logf(red[0]);
            stat[1] = l[y];
        }
        __syncthreads();
        const float lse = stat[0];
        loss += lse - stat[1];
        if (yq) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) l[i] = (expf(l[i] - lse) - (i == y ? 1.f : 0.f)) / (float)B;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && loss_out) loss_out[b] = loss;
}

// Adam on the flat float32 parameters; the float16 copy is refreshed from the result.
__global__ void k_adam(float* __restrict__ p, __half* __restrict__ p16, const float* __restrict__ g,
                       float* __restrict__ m, float* __restrict__ v, size_t n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = pi;
        p16[i] = __float2half_rn(pi);
    }
}

__global__ void k_to_half(const float* __restrict__ p, __half* __restrict__ p16, size_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        p16[i] = __float2half_rn(p[i]);
}

// Counter-based initialisation (SplitMix64 of the index and seed -> uniform in [-a, a)).
__global__ void k_init_uniform(float* __restrict__ p, size_t n, unsigned long long seed, float a) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        unsigned long long z = seed + (unsigned long long)i * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        const float u = (float)(z >> 40) * (1.0f / 16777216.0f);
        p[i] = (2.f * u - 1.f) * a;
    }
}

// ------------------------------------------------------------------ top-k joint bins
// score(q, d) = log_softmax(lq)[q] + log_softmax(ld)[d]; the k best joint bins q * nd + d of each
// sample, best first; ties to the lower bin.  Bins whose score is NaN are left out, and what is then
// missing of the k is (0x7fffffff, -inf).

// ln sum exp of both heads' logits into *lse_q, *lse_d and d - lse_d into dls, by the first kT threads of
// the block in a fixed order (every thread of the block takes part in the barriers).
__device__ void joint_log_norms(const float* q, int nq, const float* d, int nd, float* rv, float* lse_q, float* lse_d,
                                float* dls) {
    const int t = threadIdx.x;
    for (int head = 0; head < 2; ++head) {
        const float* l = head ? d : q;
        const int n = head ? nd : nq;
        float m = -INFINITY;
        if (t < kT) {
            for (int i = t; i < n; i += kT) m = fmaxf(m, l[i]);
            rv[t] = m;
        }
        __syncthreads();
        for (int st = kT / 2; st > 0; st >>= 1) {
            if (t < st) rv[t] = fmaxf(rv[t], rv[t + st]);
            __syncthreads();
        }
        m = rv[0];
        __syncthreads();
        if (t < kT) {
            float s = 0.f;
            for (int i = t; i < n; i += kT) s += expf(l[i] - m);
            rv[t] = s;
        }
        __syncthreads();
        for (int st = kT / 2; st > 0; st >>= 1) {
            if (t < st) rv[t] += rv[t + st];
            __syncthreads();
        }
        if (t == 0) *(head ? lse_d : lse_q) = m + logf(rv[0]);
        __syncthreads();
    }
    for (int i = t; i < nd; i += blockDim.x) dls[i] = d[i] - *lse_d;
    __syncthreads();
}

// Selection and sort, one block per sample: a radix selection finds the k-th largest score (each pass
// histograms kSelBits more bits of the order-preserving integer form of the scores, starting below
// the bits they all share), the k bins are compacted into shared memory and sorted there by (score,
// bin) with a bitonic network, whose steps inside a warp's own 64 entries need no block barrier.
// Bound by the sort's shared-memory passes: 0.5 log2(k)^2 of them, against one pass over all nq nd
// scores for every bin picked before (k = 4096 of 18,432, 256 samples: 54.2 ms).
constexpr int kTopT = 1024, kSelBits = 11;
static_assert(kTopT == 32 * 32 && kT >= 32, "a warp scans the warps' counts");
constexpr int kTopMaxK = 32768, kTopMaxBins = 65536;   // 6 bytes per sorted entry in shared memory; 16-bit bins

// a before b: larger score first, then the lower bin
__device__ __forceinline__ bool topk_before(uint32_t ka, uint32_t ia, uint32_t kb, uint32_t ib) {
    return ka > kb || (ka == kb && ia < ib);
}

__global__ void __launch_bounds__(kTopT) k_topk_joint(const float* __restrict__ lq, int nq, const float* __restrict__ ld,
                                                      int nd, int k, int n2, int* __restrict__ bins,
                                                      float* __restrict__ scores) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    uint32_t* key = reinterpret_cast<uint32_t*>(sm_raw);             // [n2]
    uint16_t* idx = reinterpret_cast<uint16_t*>(key + n2);           // [n2]
    __shared__ uint32_t hist[1 << kSelBits];
    __shared__ float rv[kT], dls[64], lse_q, lse_d;
    __shared__ uint32_t s_min, s_max, s_valid, s_bin, s_above, s_taken;
    const int t = threadIdx.x, lane = t & 31;
    const float* q = lq + (size_t)blockIdx.x * nq;
    const float* d = ld + (size_t)blockIdx.x * nd;
    if (t == 0) { s_min = 0xffffffffu; s_max = 0u; s_valid = 0u; s_taken = 0u; }
    joint_log_norms(q, nq, d, nd, rv, &lse_q, &lse_d, dls);
    const float lse = lse_q;
    // order-preserving integer of a score (-0 as +0); 0 for NaN, which is below every score's
    auto ord = [&](float v) -> uint32_t {
        const uint32_t u = __float_as_uint(v + 0.f);
        return v != v ? 0u : (u & 0x80000000u) ? ~u : u | 0x80000000u;
    };
    {
        uint32_t lo = 0xffffffffu, hi = 0u, c = 0;
        for (int i = t; i < nq; i += kTopT) {
            const float base = q[i] - lse;
            for (int e = 0; e < nd; ++e) {
                const uint32_t o = ord(base + dls[e]);
                if (o) { lo = min(lo, o); hi = max(hi, o); ++c; }
            }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) { atomicMin(&s_min, lo); atomicMax(&s_max, hi); atomicAdd(&s_valid, c); }
    }
    __syncthreads();
    const uint32_t valid = s_valid;
    const uint32_t need = valid < (uint32_t)k ? valid : (uint32_t)k;
    // scores with (o >> shift) > prefix are all taken; of those equal to it, the next `left`
    uint32_t prefix = 0, left = 0;
    int shift = 32;
    bool split = need < valid;   // some valid scores stay out
    if (split) {
        const uint32_t diff = s_min ^ s_max;
        shift = diff ? 32 - __clz(diff) : 0;
        prefix = shift < 32 ? s_max >> shift : 0u;
        left = need;
        while (shift > 0) {
            const int w = min(shift, kSelBits), ns = shift - w;
            for (int i = t; i < (1 << kSelBits); i += kTopT) hist[i] = 0;
            __syncthreads();
            for (int i = t; i < nq; i += kTopT) {
                const float base = q[i] - lse;
                for (int e = 0; e < nd; ++e) {
                    const uint32_t o = ord(base + dls[e]);
                    if (o && (shift == 32 || (o >> shift) == prefix)) atomicAdd(&hist[(o >> ns) & ((1u << w) - 1u)], 1u);
                }
            }
            __syncthreads();
            if (t < 32) {   // the bin, from the top, in which the count reaches `left`
                uint32_t above = 0;
                for (int b0 = (1 << w) - 1; b0 >= 0; b0 -= 32) {
                    const int b = b0 - lane;
                    const uint32_t c = b >= 0 ? hist[b] : 0u;
                    uint32_t run = c;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const uint32_t v = __shfl_up_sync(0xffffffffu, run, off);
                        if (lane >= off) run += v;
                    }
                    const unsigned hit = __ballot_sync(0xffffffffu, above + run >= left);
                    if (hit) {
                        if (lane == __ffs(hit) - 1) { s_bin = (uint32_t)b; s_above = above + run - c; }
                        break;
                    }
                    above += __shfl_sync(0xffffffffu, run, 31);
                }
            }
            __syncthreads();
            prefix = (shift == 32 ? 0u : prefix << w) | s_bin;
            left -= s_above;
            shift = ns;
            const bool whole = hist[s_bin] == left;   // the bin is taken whole: no finer threshold needed
            __syncthreads();
            if (whole) { split = false; break; }
        }
    }
    // compact: everything above the threshold prefix, and the prefix's own unless only some are taken
    const bool all = need == valid && shift == 32;
    for (int i = t; i < nq; i += kTopT) {
        const float base = q[i] - lse;
        for (int e = 0; e < nd; ++e) {
            const uint32_t o = ord(base + dls[e]);
            const uint32_t top = all ? 0u : o >> shift;
            if (o && (all || top > prefix || (top == prefix && !split))) {
                const uint32_t at = atomicAdd(&s_taken, 1u);
                key[at] = o;
                idx[at] = (uint16_t)(i * nd + e);
            }
        }
    }
    __syncthreads();
    if (split) {   // equal scores at the threshold (shift = 0): the lowest bins, kTopT at a time
        uint32_t at = s_taken;   // rv is free since joint_log_norms: the warps' counts
        uint32_t* count = reinterpret_cast<uint32_t*>(rv);
        const int total = nq * nd;
        for (int j0 = 0; j0 < total && at < need; j0 += kTopT) {   // uniform over the block
            const int j = j0 + t;
            const bool tie = j < total && ord((q[j / nd] - lse) + dls[j % nd]) == prefix;
            const unsigned bal = __ballot_sync(0xffffffffu, tie);
            if (lane == 0) count[t >> 5] = __popc(bal);
            __syncthreads();
            uint32_t run = count[lane];   // kTopT / 32 = 32 warps
            const uint32_t own = run;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t v = __shfl_up_sync(0xffffffffu, run, off);
                if (lane >= off) run += v;
            }
            const uint32_t my = at + __shfl_sync(0xffffffffu, run - own, t >> 5) + __popc(bal & ((1u << lane) - 1u));
            if (tie && my < need) {
                key[my] = prefix;
                idx[my] = (uint16_t)j;
            }
            at += __shfl_sync(0xffffffffu, run, 31);
            __syncthreads();   // the counts have been read
        }
    }
    for (int i = need + t; i < n2; i += kTopT) { key[i] = 0u; idx[i] = 0xffffu; }   // after every score
    __syncthreads();
    for (int size = 2; size <= n2; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int e = t; e < n2 / 2; e += kTopT) {
                const int i = 2 * e - (e & (stride - 1)), j = i + stride;
                const uint32_t ka = key[i], kb = key[j], ia = idx[i], ib = idx[j];
                if (topk_before(ka, ia, kb, ib) != ((i & size) == 0)) {
                    key[i] = kb; key[j] = ka;
                    idx[i] = (uint16_t)ib; idx[j] = (uint16_t)ia;
                }
            }
            // the next step's pairs of a warp lie within its own 64 entries while its stride is at most 32
            if (stride > 32 || (stride == 1 && size >= 64)) __syncthreads();
            else __syncwarp();
        }
    }
    __syncthreads();
    for (int r = t; r < k; r += kTopT) {
        const bool ok = (uint32_t)r < need;
        const int j = ok ? (int)idx[r] : 0x7fffffff;
        bins[(size_t)blockIdx.x * k + r] = j;
        if (scores) scores[(size_t)blockIdx.x * k + r] = ok ? (q[j / nd] - lse) + dls[j % nd] : -INFINITY;
    }
}

// Few picks go faster by k_topk_joint_scan, which has no selection and no sort: us for 256 samples, scan against
// sort, 1,200 bins k = 4: 8 and 23, k = 8: 16 and 23; 6,000 bins k = 1: 6 and 20, k = 3: 16 and 21; 18,432 bins k = 1: 13 and 48.
bool scan_is_short(int k, long long bins) { return k <= 3 || (k <= 8 && bins <= 2048); }

// Any nq, nd and k: one pass over the scores for each of the k picks (a sort of more than kTopMaxK
// entries or of bins beyond 16 bits does not fit in shared memory).
__global__ void __launch_bounds__(kT) k_topk_joint_scan(const float* __restrict__ lq, int nq,
                                                        const float* __restrict__ ld, int nd, int k,
                                                        int* __restrict__ bins, float* __restrict__ scores) {
    const int b = blockIdx.x;
    const float* q = lq + (size_t)b * nq;
    const float* d = ld + (size_t)b * nd;
    __shared__ float rv[kT];
    __shared__ int ri[kT];
    __shared__ float lse_q, lse_d;
    __shared__ float dls[64];
    joint_log_norms(q, nq, d, nd, rv, &lse_q, &lse_d, dls);
    const int total = nq * nd;
    int last = -1;
    float last_v = INFINITY;
    for (int r = 0; r < k; ++r) {
        float bv = -INFINITY;
        int bi = 0x7fffffff;
        for (int j = threadIdx.x; j < total; j += blockDim.x) {
            const int qi = j / nd, di = j - (j / nd) * nd;
            const float v = q[qi] - lse_q + dls[di];
            // strictly after the previous pick in (value desc, index asc) order
            const bool after = (v < last_v) || (v == last_v && j > last);
            if (after && (v > bv || (v == bv && j < bi))) {
                bv = v;
                bi = j;
            }
        }
        rv[threadIdx.x] = bv;
        ri[threadIdx.x] = bi;
        __syncthreads();
        for (int st = blockDim.x / 2; st > 0; st >>= 1) {
            if (threadIdx.x < st) {
                const float v2 = rv[threadIdx.x + st];
                const int i2 = ri[threadIdx.x + st];
                if (v2 > rv[threadIdx.x] || (v2 == rv[threadIdx.x] && i2 < ri[threadIdx.x])) {
                    rv[threadIdx.x] = v2;
                    ri[threadIdx.x] = i2;
                }
            }
            __syncthreads();
        }
        last = ri[0];
        last_v = rv[0];
        if (threadIdx.x == 0) {
            bins[(size_t)b * k + r] = last;
            if (scores) scores[(size_t)b * k + r] = last_v;
        }
        __syncthreads();
    }
}

int grid_for(size_t n) {
    size_t g = (n + kT - 1) / kT;
    return (int)(g < 65535 * 4 ? (g < 1 ? 1 : g) : 65535 * 4);
}

}  // namespace

struct bioem_cnn {
    bioem_ctx* ctx;
    int device;            // bioem_cnn_free uses these, never the (possibly destroyed) context
    cudaStream_t stream;
    int S, C, n_q, n_d, max_batch, down, n_in;
    Layer layers[kLayers];
    size_t n_params, F;
    float* d_p;        // float32 master parameters
    __half* d_p16;     // float16 copy used by the passes
    float* d_g;        // gradients
    float* d_m;        // Adam moments
    float* d_v;
    long long step;
    float* d_act;      // activations: x0 (input) then every layer output
    float* d_gact;     // their gradients
    size_t act_per_sample;
    float* d_lq;       // [max_batch][n_q]
    float* d_ld;       // [max_batch][n_d]
    float* d_loss;     // [max_batch]
    float* d_part;     // the weight-gradient blocks' partial sums of one layer
};

namespace {

template <class T>
int cnn_alloc(bioem_ctx* ctx, T** p, size_t n) {
    if (cudaMalloc((void**)p, sizeof(T) * (n ? n : 1)) != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return bioem_set_error(ctx, BIOEM_ERR_OOM, "network allocation of %zu bytes", sizeof(T) * n);
    }
    return BIOEM_OK;
}

int check(bioem_ctx* ctx, const char* what) { return bioem_check_cuda(ctx, cudaGetLastError(), what); }

struct HeadOffsets {
    size_t wq, bq, wd, bd;
};

HeadOffsets heads(const bioem_cnn* n) {
    HeadOffsets h;
    h.wq = n->layers[kLayers - 1].b_off + n->C;
    h.bq = h.wq + (size_t)n->n_q * n->F;
    h.wd = h.bq + n->n_q;
    h.bd = h.wd + (size_t)n->n_d * n->F;
    return h;
}

int prepare_input(bioem_cnn* n, const float* d_images, int B) {
    k_downsample_norm<<<B, kT, 0, n->ctx->stream>>>(d_images, n->n_in, n->down, n->d_act);
    n->ctx->n_launches++;
    return check(n->ctx, "cnn input");
}

// Output channels per thread: 16 while that leaves at least three blocks per SM, else 8, else 4.
int conv_co(const bioem_ctx* ctx, long long n_tasks, int channels) {
    int co = 16;
    while (co > 4 && (n_tasks + kConvT - 1) / kConvT * ((channels + co - 1) / co) < 3ll * ctx->num_sms) co /= 2;
    return co;
}

template <int CO, bool BWD>
void conv_launch(bioem_cnn* n, const Layer& Ly, const float* in, const float* mask, int groups, long long n_tasks,
                 float* out) {
    const int ci = BWD ? Ly.cout : Ly.cin, co = BWD ? Ly.cin : Ly.cout;   // channels read and written
    const dim3 grid((unsigned)((n_tasks + kConvT - 1) / kConvT), (co + CO - 1) / CO);
    const size_t sm = sizeof(float) * ci * 9 * CO;   // at most 64 * 9 * 16 * 4 = 36 KB
    const __half *w = n->d_p16 + Ly.w_off, *b = n->d_p16 + Ly.b_off;
    cudaStream_t st = n->ctx->stream;
    const bool vec = Ly.hout % XT == 0;
#define CONV_ARGS grid, kConvT, sm, st >>> (in, w, b, mask, ci, co, Ly.hin, Ly.hout, groups, n_tasks, out)
    if (Ly.stride == 1) {
        if (vec) k_conv<CO, 1, true, BWD><<<CONV_ARGS;
        else k_conv<CO, 1, false, BWD><<<CONV_ARGS;
    } else if constexpr (!BWD) {
        if (vec) k_conv<CO, 2, true, BWD><<<CONV_ARGS;
        else k_conv<CO, 2, false, BWD><<<CONV_ARGS;
    }
#undef CONV_ARGS
    n->ctx->n_launches++;
}

// Forward: in -> out.  BWD (stride 1): the output's gradient in -> the input's gradient out, masked.
template <bool BWD>
void launch_conv(bioem_cnn* n, const Layer& Ly, const float* in, const float* mask, int B, float* out) {
    const int groups = (Ly.hout + XT - 1) / XT;
    const long long n_tasks = (long long)B * Ly.hout * groups;
    switch (conv_co(n->ctx, n_tasks, BWD ? Ly.cin : Ly.cout)) {
        case 16: conv_launch<16, BWD>(n, Ly, in, mask, groups, n_tasks, out); break;
        case 8: conv_launch<8, BWD>(n, Ly, in, mask, groups, n_tasks, out); break;
        default: conv_launch<4, BWD>(n, Ly, in, mask, groups, n_tasks, out); break;
    }
}

void launch_conv_bwd_data(bioem_cnn* n, const Layer& Ly, const float* gout, const float* mask, int B, float* din) {
    if (Ly.stride == 1) return launch_conv<true>(n, Ly, gout, mask, B, din);
    const int groups = (Ly.hout + XT - 1) / XT;
    const long long n_tasks = (long long)B * Ly.hout * groups;
    const dim3 grid((unsigned)((n_tasks + kConvT - 1) / kConvT), (Ly.cin + CI2 - 1) / CI2);
    const size_t sm = sizeof(float) * Ly.cout * 9 * CI2;
    const __half* w = n->d_p16 + Ly.w_off;
    if (Ly.hout % XT == 0)
        k_conv_bwd_data2<true><<<grid, kConvT, sm, n->ctx->stream>>>(gout, w, mask, Ly.cin, Ly.cout, Ly.hin, Ly.hout,
                                                                     groups, n_tasks, din);
    else
        k_conv_bwd_data2<false><<<grid, kConvT, sm, n->ctx->stream>>>(gout, w, mask, Ly.cin, Ly.cout, Ly.hin, Ly.hout,
                                                                      groups, n_tasks, din);
    n->ctx->n_launches++;
}

// Weight-gradient blocks per channel block: two per SM over all of them, at most one per tile.
int wgrad_blocks(const bioem_ctx* ctx, long long units, int channel_blocks) {
    const long long most = 2ll * ctx->num_sms / channel_blocks > 0 ? 2ll * ctx->num_sms / channel_blocks : 1;
    return (int)(units < most ? units : most);
}

template <int STRIDE, int GW>
int conv_wgrad_launch(bioem_ctx* ctx, const Layer& Ly, const float* gout, const float* in, int B, int channel_blocks,
                      float* part, int* blocks) {
    using W = WgTile<STRIDE, GW>;
    const long long tiles = (long long)((Ly.hout + W::WR - 1) / W::WR) * ((Ly.hout + GW - 1) / GW);
    *blocks = wgrad_blocks(ctx, B * tiles, channel_blocks);
    auto kern = Ly.hout % 4 == 0 ? k_conv_wgrad<STRIDE, GW, true> : k_conv_wgrad<STRIDE, GW, false>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W::SMEM) != cudaSuccess)
        return bioem_check_cuda(ctx, cudaGetLastError(), "cnn shared memory");
    kern<<<dim3(*blocks, channel_blocks), kWgT, W::SMEM, ctx->stream>>>(gout, in, B, Ly.cin, Ly.cout, Ly.hin, Ly.hout, part);
    return BIOEM_OK;
}

int launch_conv_wgrad(bioem_cnn* n, const Layer& Ly, const float* gout, const float* in, int B, float* g) {
    bioem_ctx* ctx = n->ctx;
    int blocks = 0, rc = BIOEM_OK;
    if (Ly.cin == 1 && Ly.stride == 1) {
        const int gw = Ly.hout < kWgX ? (Ly.hout + 3) / 4 * 4 : kWgX;
        const long long tiles = (long long)((Ly.hout + kW1Rows - 1) / kW1Rows) * ((Ly.hout + gw - 1) / gw);
        blocks = wgrad_blocks(ctx, B * tiles, 1);
        const size_t sm = sizeof(float) * (kW1Rows + 2) * (gw + 4);
        k_conv_wgrad1<<<dim3(blocks, (Ly.cout + kW1C - 1) / kW1C), kWgT, sm, ctx->stream>>>(gout, in, B, Ly.cout, Ly.hout,
                                                                                        n->d_part);
    } else {
        const int cb = ((Ly.cout + kWgC - 1) / kWgC) * ((Ly.cin + kWgC - 1) / kWgC);
        // the narrowest tile that holds an output row, at most kWgX columns
#define WG(S, W) conv_wgrad_launch<S, W>(ctx, Ly, gout, in, B, cb, n->d_part, &blocks)
#define WG_S(S) (Ly.hout <= 8 ? WG(S, 8) : Ly.hout <= 16 ? WG(S, 16) : Ly.hout <= 32 ? WG(S, 32) : WG(S, kWgX))
        rc = Ly.stride == 1 ? WG_S(1) : WG_S(2);
#undef WG_S
#undef WG
        if (rc) return rc;
    }
    const int n_w = Ly.cout * Ly.cin * 9, total = n_w + Ly.cout;
    k_conv_wgrad_sum<<<(total + 31) / 32, kT, 0, ctx->stream>>>(n->d_part, blocks, n_w, total, g + Ly.w_off,
                                                               g + Ly.b_off);
    ctx->n_launches += 2;
    return BIOEM_OK;
}

// Forward from the prepared input (x0 at d_act) of B samples; logits into d_lq, d_ld.
int forward(bioem_cnn* n, int B) {
    bioem_ctx* ctx = n->ctx;
    cudaStream_t st = ctx->stream;
    for (int l = 0; l < kLayers; ++l) {
        const Layer& Ly = n->layers[l];
        const float* in = n->d_act + Ly.in_off * B;
        float* out = n->d_act + Ly.out_off * B;
        launch_conv<false>(n, Ly, in, nullptr, B, out);
    }
    const float* feat = n->d_act + n->layers[kLayers - 1].out_off * B;
    const HeadOffsets h = heads(n);
    const HeadFwd op{feat, n->d_p16 + h.wq, n->d_p16 + h.bq, n->d_p16 + h.wd, n->d_p16 + h.bd, n->d_lq, n->d_ld,
                     B, n->n_q, n->n_d, (int)n->F};
    const dim3 g((n->n_q + n->n_d + 63) / 64, (B + 63) / 64);
    k_gemm<64, 64, 8, 4><<<g, kGemmT, 0, st>>>(op, (int)n->F, (int)n->F);
    ctx->n_launches++;
    return check(ctx, "cnn forward");
}

// Loss and every parameter gradient (into g) for B labelled samples, after forward().
int backward(bioem_cnn* n, const int* d_yq, const int* d_yd, int B, float* g) {
    bioem_ctx* ctx = n->ctx;
    cudaStream_t st = ctx->stream;
    k_softmax_ce<<<B, kT, 0, st>>>(n->d_lq, n->n_q, n->d_ld, n->n_d, d_yq, d_yd, B, n->d_loss);
    const Layer& last = n->layers[kLayers - 1];
    const float* feat = n->d_act + last.out_off * B;
    const HeadOffsets h = heads(n);
    const int F = (int)n->F;
    // head weights gW[o][f] = sum_b glogit[b][o] feat[b][f]; biases: column sums
    const HeadGradW gw{n->d_lq, n->d_ld, feat, g + h.wq, g + h.wd, B, n->n_q, n->n_d, F};
    k_gemm<64, 64, 8, 4><<<dim3((F + 63) / 64, (n->n_q + n->n_d + 63) / 64), kGemmT, 0, st>>>(gw, B, B);
    k_colsum<<<(n->n_q + 31) / 32 + (n->n_d + 31) / 32, kT, 0, st>>>(n->d_lq, n->n_q, n->d_ld, n->n_d, B, g + h.bq,
                                                                   g + h.bd);
    // feature gradient gfeat[b][f] = sum_o glq[b][o] Wq[o][f] + sum_o gld[b][o] Wd[o][f]: few tiles and a long k,
    // so k is split into about six tiles per SM; the parts lie where the first layer's output gradient is
    // written later (C S^2 B floats, at least kFeatSplits F B)
    float* gfeat = n->d_gact + last.out_off * B;
    const HeadGradX gx{n->d_lq, n->d_p16 + h.wq, n->d_gact + n->layers[0].out_off * B, B, n->n_q, F};
    const dim3 tiles((F + 63) / 64, (B + 63) / 64);
    long long splits = 6ll * ctx->num_sms / ((long long)tiles.x * tiles.y);
    splits = splits < 1 ? 1 : splits > kFeatSplits ? kFeatSplits : splits;
    const int kps = (int)(((n->n_q + splits - 1) / splits + KT - 1) / KT * KT);
    splits = (n->n_q + kps - 1) / kps;
    k_gemm<64, 64, 8, 4><<<dim3(tiles.x, tiles.y, (unsigned)splits), kGemmT, 0, st>>>(gx, kps, n->n_q);
    k_feat_grad<<<grid_for((size_t)B * F), kT, 0, st>>>(gx.part, (int)splits, B, F, n->d_ld, n->d_p16 + h.wd, n->n_d, feat,
                                                        gfeat);
    ctx->n_launches += 5;
    // conv layers, last to first
    for (int l = kLayers - 1; l >= 0; --l) {
        const Layer& Ly = n->layers[l];
        const float* gout = n->d_gact + Ly.out_off * B;   // already through the layer's ReLU
        const float* in = n->d_act + Ly.in_off * B;
        const int rc = launch_conv_wgrad(n, Ly, gout, in, B, g);
        if (rc) return rc;
        if (l > 0) launch_conv_bwd_data(n, Ly, gout, in, B, n->d_gact + Ly.in_off * B);
    }
    return check(ctx, "cnn backward");
}

}  // namespace

extern "C" {

int bioem_cnn_create(bioem_ctx* ctx, int image_px, int downsample, int channels, int n_qbins, int n_dbins,
                     int max_batch, unsigned long long seed, bioem_cnn** out) {
    if (!ctx || !out) return BIOEM_ERR_INVALID_ARG;
    *out = nullptr;
    if (downsample < 1 || image_px % downsample || (image_px / downsample) % 8 || image_px / downsample < 8 ||
        channels < 1 || channels > 64 || n_qbins < 1 || n_dbins < 1 || n_dbins > 64 || max_batch < 1)
        return bioem_set_error(ctx, BIOEM_ERR_INVALID_ARG, "cnn_create: bad shape");
    if (cudaSetDevice(ctx->device) != cudaSuccess) return bioem_set_error(ctx, BIOEM_ERR_CUDA, "cudaSetDevice");
    bioem_cnn* n = new (std::nothrow) bioem_cnn();
    if (!n) return BIOEM_ERR_OOM;
    n->ctx = ctx;
    n->device = ctx->device;
    n->stream = ctx->stream;
    n->n_in = image_px;
    n->down = downsample;
    n->S = image_px / downsample;
    n->C = channels;
    n->n_q = n_qbins;
    n->n_d = n_dbins;
    n->max_batch = max_batch;
    const int strides[kLayers] = {1, 2, 1, 2, 1, 2};
    size_t poff = 0, aoff = (size_t)n->S * n->S;   // x0 occupies the first S^2 per sample
    int h = n->S, cin = 1;
    for (int l = 0; l < kLayers; ++l) {
        Layer& Ly = n->layers[l];
        Ly.cin = cin;
        Ly.cout = channels;
        Ly.stride = strides[l];
        Ly.hin = h;
        Ly.hout = h / strides[l];
        Ly.w_off = poff;
        poff += (size_t)channels * cin * 9;
        Ly.b_off = poff;
        poff += channels;
        Ly.in_off = (l == 0) ? 0 : n->layers[l - 1].out_off;
        Ly.out_off = aoff;
        aoff += (size_t)channels * Ly.hout * Ly.hout;
        h = Ly.hout;
        cin = channels;
    }
    n->F = (size_t)channels * h * h;
    n->n_params = poff + (size_t)n_qbins * n->F + n_qbins + (size_t)n_dbins * n->F + n_dbins;
    n->act_per_sample = aoff;
    int rc = cnn_alloc(ctx, &n->d_p, n->n_params);
    if (!rc) rc = cnn_alloc(ctx, &n->d_p16, n->n_params);
    if (!rc) rc = cnn_alloc(ctx, &n->d_g, n->n_params);
    if (!rc) rc = cnn_alloc(ctx, &n->d_m, n->n_params);
    if (!rc) rc = cnn_alloc(ctx, &n->d_v, n->n_params);
    if (!rc) rc = cnn_alloc(ctx, &n->d_act, n->act_per_sample * max_batch);
    if (!rc) rc = cnn_alloc(ctx, &n->d_gact, n->act_per_sample * max_batch);
    if (!rc) rc = cnn_alloc(ctx, &n->d_lq, (size_t)max_batch * n_qbins);
    if (!rc) rc = cnn_alloc(ctx, &n->d_ld, (size_t)max_batch * n_dbins);
    if (!rc) rc = cnn_alloc(ctx, &n->d_loss, (size_t)max_batch);
    if (!rc) rc = cnn_alloc(ctx, &n->d_part, 2 * (size_t)ctx->num_sms * ((size_t)channels * channels * 9 + channels));
    if (rc) {
        bioem_cnn_free(n);
        return rc;
    }
    cudaStream_t st = ctx->stream;
    // uniform He-style initialisation per tensor: a = sqrt(6 / fan_in); biases zero
    for (int l = 0; l < kLayers; ++l) {
        const Layer& Ly = n->layers[l];
        const size_t nw = (size_t)Ly.cout * Ly.cin * 9;
        k_init_uniform<<<grid_for(nw), kT, 0, st>>>(n->d_p + Ly.w_off, nw, seed + 1000003ull * l,
                                                    sqrtf(6.f / (9.f * Ly.cin)));
        cudaMemsetAsync(n->d_p + Ly.b_off, 0, sizeof(float) * Ly.cout, st);
    }
    const HeadOffsets hd = heads(n);
    k_init_uniform<<<grid_for((size_t)n_qbins * n->F), kT, 0, st>>>(n->d_p + hd.wq, (size_t)n_qbins * n->F, seed + 77ull,
                                                                     sqrtf(3.f / (float)n->F));
    k_init_uniform<<<grid_for((size_t)n_dbins * n->F), kT, 0, st>>>(n->d_p + hd.wd, (size_t)n_dbins * n->F, seed + 78ull,
                                                                     sqrtf(3.f / (float)n->F));
    cudaMemsetAsync(n->d_p + hd.bq, 0, sizeof(float) * n_qbins, st);
    cudaMemsetAsync(n->d_p + hd.bd, 0, sizeof(float) * n_dbins, st);
    cudaMemsetAsync(n->d_m, 0, sizeof(float) * n->n_params, st);
    cudaMemsetAsync(n->d_v, 0, sizeof(float) * n->n_params, st);
    k_to_half<<<grid_for(n->n_params), kT, 0, st>>>(n->d_p, n->d_p16, n->n_params);
    ctx->n_launches += kLayers + 3;
    rc = check(ctx, "cnn init");
    if (rc) {
        bioem_cnn_free(n);
        return rc;
    }
    *out = n;
    return BIOEM_OK;
}

long long bioem_cnn_num_params(const bioem_cnn* n) { return n ? (long long)n->n_params : -1; }

int bioem_cnn_set_params(bioem_cnn* n, const float* d_params) {
    if (!n || !d_params) return BIOEM_ERR_INVALID_ARG;
    cudaSetDevice(n->ctx->device);
    cudaStream_t st = n->ctx->stream;
    cudaError_t e = cudaMemcpyAsync(n->d_p, d_params, sizeof(float) * n->n_params, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return bioem_check_cuda(n->ctx, e, "set params");
    k_to_half<<<grid_for(n->n_params), kT, 0, st>>>(n->d_p, n->d_p16, n->n_params);
    n->ctx->n_launches++;
    cudaMemsetAsync(n->d_m, 0, sizeof(float) * n->n_params, st);
    cudaMemsetAsync(n->d_v, 0, sizeof(float) * n->n_params, st);
    n->step = 0;
    return check(n->ctx, "set params");
}

int bioem_cnn_get_params(bioem_cnn* n, float* d_params) {
    if (!n || !d_params) return BIOEM_ERR_INVALID_ARG;
    cudaSetDevice(n->ctx->device);
    return bioem_check_cuda(n->ctx, cudaMemcpyAsync(d_params, n->d_p, sizeof(float) * n->n_params,
                                                    cudaMemcpyDeviceToDevice, n->ctx->stream), "get params");
}

int bioem_cnn_forward(bioem_cnn* n, const float* d_images, int B, float* d_logits_q, float* d_logits_d) {
    if (!n || !d_images || B < 1 || B > n->max_batch) return BIOEM_ERR_INVALID_ARG;
    cudaSetDevice(n->ctx->device);
    int rc = prepare_input(n, d_images, B);
    if (!rc) rc = forward(n, B);
    cudaStream_t st = n->ctx->stream;
    if (!rc && d_logits_q)
        rc = bioem_check_cuda(n->ctx, cudaMemcpyAsync(d_logits_q, n->d_lq, sizeof(float) * B * n->n_q,
                                                      cudaMemcpyDeviceToDevice, st), "logits");
    if (!rc && d_logits_d)
        rc = bioem_check_cuda(n->ctx, cudaMemcpyAsync(d_logits_d, n->d_ld, sizeof(float) * B * n->n_d,
                                                      cudaMemcpyDeviceToDevice, st), "logits");
    return rc;
}

int bioem_cnn_gradients(bioem_cnn* n, const float* d_images, const int* d_label_q, const int* d_label_d, int B,
                        float* d_grads, float* d_loss) {
    if (!n || !d_images || !d_label_q || !d_label_d || B < 1 || B > n->max_batch) return BIOEM_ERR_INVALID_ARG;
    cudaSetDevice(n->ctx->device);
    int rc = prepare_input(n, d_images, B);
    if (!rc) rc = forward(n, B);
    if (!rc) rc = backward(n, d_label_q, d_label_d, B, d_grads ? d_grads : n->d_g);
    cudaStream_t st = n->ctx->stream;
    if (!rc && d_loss)
        rc = bioem_check_cuda(n->ctx, cudaMemcpyAsync(d_loss, n->d_loss, sizeof(float) * B, cudaMemcpyDeviceToDevice, st),
                              "loss");
    return rc;
}

int bioem_cnn_train_step(bioem_cnn* n, const float* d_images, const int* d_label_q, const int* d_label_d, int B,
                         float lr, float* d_loss) {
    int rc = bioem_cnn_gradients(n, d_images, d_label_q, d_label_d, B, nullptr, d_loss);
    if (rc) return rc;
    n->step++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)n->step), c2 = 1.f - powf(b2, (float)n->step);
    k_adam<<<grid_for(n->n_params), kT, 0, n->ctx->stream>>>(n->d_p, n->d_p16, n->d_g, n->d_m, n->d_v, n->n_params, lr,
                                                             b1, b2, 1e-8f, c1, c2);
    n->ctx->n_launches++;
    return check(n->ctx, "adam");
}

int bioem_propose(bioem_cnn* n, const float* d_images, int n_img, int k, int* d_bins, float* d_scores) {
    if (!n || !d_images || n_img < 0 || k < 1 || k > n->n_q * n->n_d || !d_bins) return BIOEM_ERR_INVALID_ARG;
    cudaSetDevice(n->ctx->device);
    const long long n_bins = (long long)n->n_q * n->n_d;
    const bool sorted = k <= kTopMaxK && n_bins <= kTopMaxBins && !scan_is_short(k, n_bins);
    int n2 = 64;   // entries of the sorting network: a power of two, at least a warp's 64
    while (sorted && n2 < k) n2 *= 2;
    const size_t sm = (size_t)n2 * 6;
    // the limit belongs to the function on this device, not to this call: the same value from every caller, so
    // that one on another thread cannot lower it before the launch
    if (sorted && cudaFuncSetAttribute(k_topk_joint, cudaFuncAttributeMaxDynamicSharedMemorySize, 6 * kTopMaxK) != cudaSuccess)
        return bioem_check_cuda(n->ctx, cudaGetLastError(), "top-k shared memory");
    for (int b0 = 0; b0 < n_img; b0 += n->max_batch) {
        const int B = n_img - b0 < n->max_batch ? n_img - b0 : n->max_batch;
        int rc = prepare_input(n, d_images + (size_t)b0 * n->n_in * n->n_in, B);
        if (!rc) rc = forward(n, B);
        if (rc) return rc;
        int* bins = d_bins + (size_t)b0 * k;
        float* scores = d_scores ? d_scores + (size_t)b0 * k : nullptr;
        if (sorted)
            k_topk_joint<<<B, kTopT, sm, n->ctx->stream>>>(n->d_lq, n->n_q, n->d_ld, n->n_d, k, n2, bins, scores);
        else
            k_topk_joint_scan<<<B, kT, 0, n->ctx->stream>>>(n->d_lq, n->n_q, n->d_ld, n->n_d, k, bins, scores);
        n->ctx->n_launches++;
        rc = check(n->ctx, "propose");
        if (rc) return rc;
    }
    return BIOEM_OK;
}

void bioem_cnn_free(bioem_cnn* n) {
    if (!n) return;
    cudaSetDevice(n->device);
    cudaStreamSynchronize(n->stream);
    cudaFree(n->d_p);
    cudaFree(n->d_p16);
    cudaFree(n->d_g);
    cudaFree(n->d_m);
    cudaFree(n->d_v);
    cudaFree(n->d_act);
    cudaFree(n->d_gact);
    cudaFree(n->d_lq);
    cudaFree(n->d_ld);
    cudaFree(n->d_loss);
    cudaFree(n->d_part);
    cudaGetLastError();
    delete n;
}

}  // extern "C"

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
constexpr int kFeatSplits = 4;   // k splits of the feature gradient (its parts need F kFeatSplits <= C S^2 = 64 F)

struct Layer {
    int cin, cout, stride, hin, hout;
    size_t w_off, b_off;     // offsets in the flat parameter vector
    size_t in_off, out_off;  // activation offsets (per-sample element counts are cin*hin^2, cout*hout^2)
};

// ------------------------------------------------------------------ input preparation
// out[b][y][x] = standardised 2x2 average of img[b]; per image: zero mean, unit variance over S^2.
__global__ void __launch_bounds__(kT) k_downsample_norm(const float* __restrict__ img, int n_in, int down,
                                                        float* __restrict__ out) {
    const int b = blockIdx.x;
    const int S = n_in / down;
    const float* src = img + (size_t)b * n_in * n_in;
    float* dst = out + (size_t)b * S * S;
    __shared__ double r1[kT], r2[kT];
    double s1 = 0.0, s2 = 0.0;
    for (int i = threadIdx.x; i < S * S; i += blockDim.x) {
        const int y = i / S, x = i - (i / S) * S;
        float v = 0.f;
        for (int dy = 0; dy < down; ++dy)
            for (int dx = 0; dx < down; ++dx) v += src[(y * down + dy) * n_in + x * down + dx];
        v *= 1.0f / (float)(down * down);
        dst[i] = v;
        s1 += v;
        s2 += (double)v * v;
    }
    r1[threadIdx.x] = s1;
    r2[threadIdx.x] = s2;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if (threadIdx.x < st) {
            r1[threadIdx.x] += r1[threadIdx.x + st];
            r2[threadIdx.x] += r2[threadIdx.x + st];
        }
        __syncthreads();
    }
    const double n = (double)S * S;
    const double mean = r1[0] / n;
    const double var = r2[0] / n - mean * mean;
    const float inv = var > 0.0 ? (float)(1.0 / sqrt(var)) : 0.f;
    const float m = (float)mean;
    for (int i = threadIdx.x; i < S * S; i += blockDim.x) dst[i] = (dst[i] - m) * inv;
}

// ------------------------------------------------------------------ convolution
// out[b][co][y][x] = ReLU(b[co] + sum_ci,ky,kx W[co][ci][ky][kx] in[b][ci][y s + ky - 1][x s + kx - 1])
//
// A thread owns XT = 4 neighbouring outputs of one row in CO output channels, so an input row segment
// loaded once serves 3 CO products per value and a weight serves XT; the products of two channels go
// out as one packed FP32 pair.  Every output is still summed in the order (ci, ky, kx) starting from
// the bias, with the taps outside the image left out, so the activations do not depend on the tiling.
// Bound by the FP32 pipe.  CO = 16 has the fewest loads per product; fewer channels per thread are
// taken where that would leave too few blocks (conv_co).  VEC: rows read as float4 with the edge
// values from the neighbouring lanes (needs output rows of whole groups of four).
constexpr int XT = 4;
constexpr int kConvT = 128;

// BWD (stride 1): the gradient of the layer's input, din[b][ci][y][x] = sum_co,ky,kx gout[b][co][y + 1 - ky]
// [x + 1 - kx] W[co][ci][ky][kx], the same sum with the channels' roles exchanged and the taps reversed
// (cin, cout are then the layer's output and input channels); no bias, and the ReLU that produced the
// layer's input (mask = that input) is applied to the result instead of in a pass of its own.
template <int CO, int STRIDE, bool VEC, bool BWD>
__global__ void __launch_bounds__(kConvT) k_conv(const float* __restrict__ in, const __half* __restrict__ W,
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
// walks over tiles of WR output rows x at most kWgX columns of one sample staged in shared memory
// (inputs with a border of zeros), four columns at a time: 144 products per 14 (stride 1) or 20 (stride 2) shared reads, against
// one read per product when each (co, ci) pair was a block of its own.  Bound by the FP32 pipe.
// Channel strides are 4 x odd floats, so the 16-byte reads of 8 neighbouring channels do not conflict.
constexpr int kWgT = 256, kWgC = 32, kWgX = 64;

__host__ __device__ constexpr int wg_rows(int stride) { return stride == 1 ? 4 : 2; }   // output rows per strip
__host__ __device__ constexpr int odd4(int n) { return ((n + 3) / 4 | 1) * 4; }          // >= n, 4 x odd
__host__ __device__ inline int wg_gw(int hout) { return hout < kWgX ? (hout + 3) / 4 * 4 : kWgX; }   // staged gout row
__host__ __device__ inline int wg_iw(int hout, int stride) { return (wg_gw(hout) * stride + 2 + 3) / 4 * 4; }
__host__ __device__ inline int wg_gch(int hout, int stride) { return odd4(wg_rows(stride) * wg_gw(hout)); }
__host__ __device__ inline int wg_ich(int hout, int stride) {
    return odd4(((wg_rows(stride) - 1) * stride + 3) * wg_iw(hout, stride));
}

template <int STRIDE>
__global__ void __launch_bounds__(kWgT, 2) k_conv_wgrad(const float* __restrict__ gout, const float* __restrict__ in,
                                                        int B, int cin, int cout, int hin, int hout,
                                                        float* __restrict__ part) {
    constexpr int WR = wg_rows(STRIDE), IR = (WR - 1) * STRIDE + 3;
    extern __shared__ __align__(16) float sm[];
    const int gw = wg_gw(hout), iw = wg_iw(hout, STRIDE), gch = wg_gch(hout, STRIDE), ich = wg_ich(hout, STRIDE);
    float* gs = sm;                   // [32 co][WR][gw]
    float* is = sm + kWgC * gch;      // [32 ci][IR][iw], column ix + 1
    const int nci = (cin + kWgC - 1) / kWgC;
    const int co0 = (int)blockIdx.y / nci * kWgC, ci0 = (int)blockIdx.y % nci * kWgC;
    const int tc = threadIdx.x & 15, to = threadIdx.x >> 4;   // ci = ci0 + tc + 16 j, co = co0 + to + 16 i
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float acc[2][2][9], sb[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int k = 0; k < 9; ++k) acc[i][j][k] = 0.f;
    const int tiles_x = (hout + gw - 1) / gw, tiles = (hout + WR - 1) / WR * tiles_x;
    const long long units = (long long)B * tiles;
    for (long long u = blockIdx.x; u < units; u += gridDim.x) {
        const int b = (int)(u / tiles), t = (int)(u - (long long)b * tiles);
        const int y0 = t / tiles_x * WR, xs = t % tiles_x * gw;
        __syncthreads();   // the previous tile has been read
        for (int r = warp; r < kWgC * WR; r += kWgT / 32) {
            const int c = r / WR, y = r - c * WR;
            const float* src = gout + (((size_t)b * cout + co0 + c) * hout + y0 + y) * hout + xs;
            const bool ok = co0 + c < cout && y0 + y < hout;
            for (int x = lane; x < gw; x += 32) gs[c * gch + y * gw + x] = ok && xs + x < hout ? __ldg(src + x) : 0.f;
        }
        for (int r = warp; r < kWgC * IR; r += kWgT / 32) {
            const int c = r / IR, y = r - c * IR;
            const int iy = y0 * STRIDE + y - 1;
            const float* src = in + (((size_t)b * cin + ci0 + c) * hin + iy) * hin;
            const bool ok = ci0 + c < cin && iy >= 0 && iy < hin;
            for (int x = lane; x < iw; x += 32) {
                const int ix = xs * STRIDE + x - 1;
                is[c * ich + y * iw + x] = ok && ix >= 0 && ix < hin ? __ldg(src + ix) : 0.f;
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int y = 0; y < WR; ++y) {
#pragma unroll 1
            for (int x0 = 0; x0 < gw; x0 += 4) {
                float g[2][4];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float4 t = *reinterpret_cast<const float4*>(gs + (to + 16 * i) * gch + y * gw + x0);
                    g[i][0] = t.x; g[i][1] = t.y; g[i][2] = t.z; g[i][3] = t.w;
                    sb[i] += (t.x + t.y) + (t.z + t.w);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky) {
                        const float* row = is + (tc + 16 * j) * ich + (y * STRIDE + ky) * iw + x0 * STRIDE;
                        float v[3 * STRIDE + 3];
#pragma unroll
                        for (int q = 0; q < STRIDE; ++q) {
                            const float4 t = *reinterpret_cast<const float4*>(row + 4 * q);
                            v[4 * q] = t.x; v[4 * q + 1] = t.y; v[4 * q + 2] = t.z; v[4 * q + 3] = t.w;
                        }
                        if constexpr (STRIDE == 1) {
                            const float2 t = *reinterpret_cast<const float2*>(row + 4);
                            v[4] = t.x; v[5] = t.y;
                        } else {
                            v[8] = row[8];
                        }
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

// The same for the first layer (one input channel, stride 1): a warp per output channel (four of a
// block's 32 in turn), its lanes over groups of four columns of a tile of 16 rows.  Bound by reading
// gout once.
constexpr int kW1Rows = 16;
__global__ void __launch_bounds__(kWgT) k_conv_wgrad1(const float* __restrict__ gout, const float* __restrict__ in,
                                                      int B, int cout, int h, float* __restrict__ part) {
    extern __shared__ __align__(16) float is[];   // [kW1Rows + 2][iw], column ix + 1
    const int gw = wg_gw(h), iw = gw + 4, q4 = gw / 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int CW = kWgC / (kWgT / 32);   // output channels per warp
    float acc[CW][10];
#pragma unroll
    for (int c = 0; c < CW; ++c)
#pragma unroll
        for (int k = 0; k < 10; ++k) acc[c][k] = 0.f;
    const int tiles_x = (h + gw - 1) / gw, tiles = (h + kW1Rows - 1) / kW1Rows * tiles_x;
    const long long units = (long long)B * tiles;
    const bool vec = h % 4 == 0;
    for (long long u = blockIdx.x; u < units; u += gridDim.x) {
        const int b = (int)(u / tiles), t = (int)(u - (long long)b * tiles);
        const int y0 = t / tiles_x * kW1Rows, xs = t % tiles_x * gw;
        __syncthreads();
        for (int i = threadIdx.x; i < (kW1Rows + 2) * iw; i += kWgT) {
            const int y = i / iw, x = i - y * iw;
            const int iy = y0 + y - 1, ix = xs + x - 1;
            is[i] = iy >= 0 && iy < h && ix >= 0 && ix < h ? __ldg(in + ((size_t)b * h + iy) * h + ix) : 0.f;
        }
        __syncthreads();
        const int rows = min(kW1Rows, h - y0);
        for (int e = lane; e < rows * q4; e += 32) {
            const int y = e / q4, x0 = (e - y * q4) * 4;
            if (xs + x0 >= h) continue;
            float v[3][6];
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
                const float* row = is + (y + ky) * iw + x0;
                const float4 t = *reinterpret_cast<const float4*>(row);
                const float2 t2 = *reinterpret_cast<const float2*>(row + 4);
                v[ky][0] = t.x; v[ky][1] = t.y; v[ky][2] = t.z; v[ky][3] = t.w; v[ky][4] = t2.x; v[ky][5] = t2.y;
            }
#pragma unroll
            for (int c = 0; c < CW; ++c) {
                const int co = blockIdx.y * kWgC + warp * CW + c;
                if (co >= cout) break;
                const float* gp = gout + (((size_t)b * cout + co) * h + y0 + y) * h + xs + x0;
                float g[4];
                if (vec) {
                    const float4 t = __ldg(reinterpret_cast<const float4*>(gp));
                    g[0] = t.x; g[1] = t.y; g[2] = t.z; g[3] = t.w;
                } else {
#pragma unroll
                    for (int x = 0; x < 4; ++x) g[x] = xs + x0 + x < h ? __ldg(gp + x) : 0.f;
                }
#pragma unroll
                for (int x = 0; x < 4; ++x) {
#pragma unroll
                    for (int k = 0; k < 9; ++k) acc[c][k] = fmaf(g[x], v[k / 3][x + k % 3], acc[c][k]);
                    acc[c][9] += g[x];
                }
            }
        }
    }
    float* o = part + (size_t)blockIdx.x * ((size_t)cout * 9 + cout);
#pragma unroll
    for (int c = 0; c < CW; ++c) {
        const int co = blockIdx.y * kWgC + warp * CW + c;
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
// buffers, the next step's operands held in registers meanwhile.  Bound by the FP32 pipe: the first
// form (4 x 4 outputs per thread, one buffer, a thread's loads a row of A apart) spent its time on
// shared-memory reads and uncoalesced loads.  The operands come from functors so that the two heads
// form one product (their columns, rows or k ranges follow one another):
//   op.a(m, k), op.b(n, k)  the operands (0 outside the product)     op.store(m, n, v)
//   OP::AK / OP::BK         true: consecutive k are adjacent in memory (else consecutive m / n)
constexpr int kGemmT = 128, KT = 16;

template <int TM, int TN, int MT, int NT, class OP>
__global__ void __launch_bounds__(kGemmT) k_gemm(const OP op, int k_per_split, int K) {
    static_assert(TM / MT * (TN / NT) == kGemmT && MT % 4 == 0 && NT % 4 == 0, "one MT x NT block per thread");
    constexpr int PA = TM * KT / kGemmT, PB = TN * KT / kGemmT;
    __shared__ __align__(16) float As[2][KT][TM + 4], Bs[2][KT][TN + 4];
    const int tn = threadIdx.x % (TN / NT), tm = threadIdx.x / (TN / NT);
    const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
    const int kb = blockIdx.z * k_per_split, ke = min(K, kb + k_per_split);
    float2 acc[MT / 2][NT];
#pragma unroll
    for (int i = 0; i < MT / 2; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j) acc[i][j] = make_float2(0.f, 0.f);
    float ra[PA], rb[PB];
    // element i of a thread's share: k-adjacent operands take 8 k x 16 rows per pass (full 32-byte
    // sectors, conflict-free transposed stores), the others a run of rows at one k
    auto at = [](bool adj, int rows, int i, int& r, int& k) {
        const int e = threadIdx.x + i * kGemmT;
        if (adj) {
            k = (e & 7) + ((e / (8 * rows)) << 3);
            r = (e >> 3) % rows;
        } else {
            r = e % rows;
            k = e / rows;
        }
    };
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < PA; ++i) {
            int r, k;
            at(OP::AK, TM, i, r, k);
            ra[i] = k0 + k < ke ? op.a(m0 + r, k0 + k) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            int r, k;
            at(OP::BK, TN, i, r, k);
            rb[i] = k0 + k < ke ? op.b(n0 + r, k0 + k) : 0.f;
        }
    };
    auto stage = [&](int buf) {
#pragma unroll
        for (int i = 0; i < PA; ++i) {
            int r, k;
            at(OP::AK, TM, i, r, k);
            As[buf][k][r] = ra[i];
        }
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            int r, k;
            at(OP::BK, TN, i, r, k);
            Bs[buf][k][r] = rb[i];
        }
    };
    fetch(kb);
    stage(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = kb; k0 < ke; k0 += KT, buf ^= 1) {
        const bool more = k0 + KT < ke;
        if (more) fetch(k0 + KT);
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
        if (more) stage(buf ^ 1);
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
            op.store(m0 + tm * MT + i, n0 + (j / 4) * (4 * TN / NT) + tn * 4 + (j & 3), (int)blockIdx.z,
                     (i & 1) ? acc[i / 2][j].y : acc[i / 2][j].x);
}

// Both heads' logits: m = sample, n = orientation bins then defocus bins, k = feature.
struct HeadFwd {
    static constexpr bool AK = true, BK = true;
    const float* feat;
    const __half *wq, *bq, *wd, *bd;
    float *lq, *ld;
    int B, nq, nd, F;
    __device__ __forceinline__ float a(int m, int k) const { return m < B ? __ldg(feat + (size_t)m * F + k) : 0.f; }
    __device__ __forceinline__ float b(int n, int k) const {
        const __half* w = n < nq ? wq + (size_t)n * F : wd + (size_t)(n - nq) * F;
        return n < nq + nd ? __half2float(w[k]) : 0.f;
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
    const float *glq, *gld, *feat;
    float *gwq, *gwd;
    int B, nq, nd, F;
    __device__ __forceinline__ float a(int m, int k) const {
        if (m >= nq + nd) return 0.f;
        return m < nq ? __ldg(glq + (size_t)k * nq + m) : __ldg(gld + (size_t)k * nd + m - nq);
    }
    __device__ __forceinline__ float b(int n, int k) const { return n < F ? __ldg(feat + (size_t)k * F + n) : 0.f; }
    __device__ __forceinline__ void store(int m, int n, int, float v) const {
        if (m >= nq + nd || n >= F) return;
        if (m < nq) gwq[(size_t)m * F + n] = v;
        else gwd[(size_t)(m - nq) * F + n] = v;
    }
};

// Feature gradients, split over k: m = sample, n = feature, k = orientation bins then defocus bins;
// part[split][m][n], summed by k_feat_grad.
struct HeadGradX {
    static constexpr bool AK = true, BK = false;
    const float *glq, *gld;
    const __half *wq, *wd;
    float* part;
    int B, nq, nd, F;
    __device__ __forceinline__ float a(int m, int k) const {
        if (m >= B) return 0.f;
        return k < nq ? __ldg(glq + (size_t)m * nq + k) : __ldg(gld + (size_t)m * nd + k - nq);
    }
    __device__ __forceinline__ float b(int n, int k) const {
        const __half* w = k < nq ? wq + (size_t)k * F : wd + (size_t)(k - nq) * F;
        return n < F ? __half2float(w[n]) : 0.f;
    }
    __device__ __forceinline__ void store(int m, int n, int z, float v) const {
        if (m < B && n < F) part[((size_t)z * B + m) * F + n] = v;
    }
};

// gfeat = the sum of the k splits, back through the ReLU whose output is feat.
__global__ void __launch_bounds__(kT) k_feat_grad(const float* __restrict__ part, int splits, size_t n,
                                                  const float* __restrict__ feat, float* __restrict__ gfeat) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        float s = 0.f;
        for (int z = 0; z < splits; ++z) s += part[(size_t)z * n + i];
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
    if (split && t < 32) {   // equal scores at the threshold (shift = 0): the lowest bins
        uint32_t at = s_taken;
        const int total = nq * nd;
        for (int j0 = 0; j0 < total && at < need; j0 += 32) {
            const int j = j0 + lane;
            const bool tie = j < total && ord((q[j / nd] - lse) + dls[j % nd]) == prefix;
            const unsigned bal = __ballot_sync(0xffffffffu, tie);
            const uint32_t my = at + __popc(bal & ((1u << lane) - 1u));
            if (tie && my < need) {
                key[my] = prefix;
                idx[my] = (uint16_t)j;
            }
            at += __popc(bal);
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

// Output channels per thread: 16 while that leaves at least four blocks per SM, else 8, else 4.
int conv_co(const bioem_ctx* ctx, long long n_tasks, int channels) {
    int co = 16;
    while (co > 4 && (n_tasks + kConvT - 1) / kConvT * ((channels + co - 1) / co) < 4ll * ctx->num_sms) co /= 2;
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

// Weight-gradient blocks: two per SM over all channel blocks, at most one per tile.
int wgrad_blocks(const bioem_ctx* ctx, long long units, int channel_blocks) {
    const long long most = 2ll * ctx->num_sms / channel_blocks > 0 ? 2ll * ctx->num_sms / channel_blocks : 1;
    return (int)(units < most ? units : most);
}

int launch_conv_wgrad(bioem_cnn* n, const Layer& Ly, const float* gout, const float* in, int B, float* g) {
    bioem_ctx* ctx = n->ctx;
    const int nco = (Ly.cout + kWgC - 1) / kWgC, nci = (Ly.cin + kWgC - 1) / kWgC;
    const int gw = wg_gw(Ly.hout), tiles_x = (Ly.hout + gw - 1) / gw;
    int blocks;
    if (Ly.cin == 1 && Ly.stride == 1) {
        blocks = wgrad_blocks(ctx, (long long)B * ((Ly.hout + kW1Rows - 1) / kW1Rows) * tiles_x, nco);
        const size_t sm = sizeof(float) * (kW1Rows + 2) * (gw + 4);
        k_conv_wgrad1<<<dim3(blocks, nco), kWgT, sm, ctx->stream>>>(gout, in, B, Ly.cout, Ly.hout, n->d_part);
    } else {
        const int wr = wg_rows(Ly.stride);
        blocks = wgrad_blocks(ctx, (long long)B * ((Ly.hout + wr - 1) / wr) * tiles_x, nco * nci);
        const size_t sm = sizeof(float) * kWgC * (size_t)(wg_gch(Ly.hout, Ly.stride) + wg_ich(Ly.hout, Ly.stride));
        auto kern = Ly.stride == 1 ? k_conv_wgrad<1> : k_conv_wgrad<2>;
        if (sm > 48 * 1024 &&
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
            return bioem_check_cuda(ctx, cudaGetLastError(), "cnn shared memory");
        kern<<<dim3(blocks, nco * nci), kWgT, sm, ctx->stream>>>(gout, in, B, Ly.cin, Ly.cout, Ly.hin, Ly.hout, n->d_part);
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
    k_gemm<128, 64, 8, 8><<<dim3((F + 63) / 64, (n->n_q + n->n_d + 127) / 128), kGemmT, 0, st>>>(gw, B, B);
    k_colsum<<<(n->n_q + 31) / 32 + (n->n_d + 31) / 32, kT, 0, st>>>(n->d_lq, n->n_q, n->d_ld, n->n_d, B, g + h.bq,
                                                                   g + h.bd);
    // feature gradient gfeat[b][f] = sum_o glq[b][o] Wq[o][f] + sum_o gld[b][o] Wd[o][f]: a short product
    // (few tiles, long k), so k is split; the parts lie where the first layer's output gradient is
    // written later (C S^2 B floats, at least kFeatSplits F B)
    float* gfeat = n->d_gact + last.out_off * B;
    const HeadGradX gx{n->d_lq, n->d_ld, n->d_p16 + h.wq, n->d_p16 + h.wd, n->d_gact + n->layers[0].out_off * B,
                       B, n->n_q, n->n_d, F};
    const int K = n->n_q + n->n_d, kps = ((K + kFeatSplits - 1) / kFeatSplits + KT - 1) / KT * KT;
    const int splits = (K + kps - 1) / kps;
    k_gemm<64, 64, 8, 4><<<dim3((F + 63) / 64, (B + 63) / 64, splits), kGemmT, 0, st>>>(gx, kps, K);
    k_feat_grad<<<grid_for((size_t)B * F), kT, 0, st>>>(gx.part, splits, (size_t)B * F, feat, gfeat);
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
    const bool sorted = k <= kTopMaxK && (long long)n->n_q * n->n_d <= kTopMaxBins;
    int n2 = 64;   // entries of the sorting network: a power of two, at least a warp's 64
    while (sorted && n2 < k) n2 *= 2;
    const size_t sm = (size_t)n2 * 6;
    if (sorted && cudaFuncSetAttribute(k_topk_joint, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
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

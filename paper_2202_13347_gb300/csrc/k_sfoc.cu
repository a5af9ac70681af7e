// SFOC descriptor kernels (Sec. 2.1 of arXiv 2202.13347).
//
// k_sfoc_steer   separable Gaussian-derivative bases (Eq. 2, 3, 5), steering
//                (Eq. 6, 7), |.| and the sum over scales -> F planes.
// k_sfoc_smooth  three parallel dilated Gaussian smoothings per channel,
//                summed, group-wise L2 normalisation and stacking, plus the
//                per-pixel sum planes used by the integral images (Eq. 14).
//
// Borders clamp to the edge in every convolution.  These two serve any radii
// and rates: they stage a 2-D tile with its clamped halo in shared memory and
// do the horizontal pass into shared planes, then the vertical pass per output
// pixel.  The paper's own parameters take the streaming forms
// k_sfoc_steer_strip and k_sfoc_smooth_strip.
#include <cuda_bf16.h>
#include <string.h>

#include <type_traits>

#include "internal.h"

namespace sfoc {

namespace {

constexpr int kTW = 32;          // output tile width (one warp across)
constexpr int kTH = 32;          // output tile height
constexpr int kThreads = 256;

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// Row stride (floats) of the smoothing input tile: room for the tile, its
// halo and the 8-wide load blocks' overrun, a multiple of 4 floats (float4
// rows) with an odd number of float4s, so that the two rows a quarter-warp
// reads in the horizontal pass fall in different banks.
__host__ __device__ inline int smooth_row_stride(int maxhal) {
    int fw = (32 + 2 * maxhal + 8 + 3) / 4 * 4;
    if ((fw / 4) % 2 == 0) fw += 4;
    return fw;
}

// even taps: t0 x[0] + sum_q t[q] (x[-q] + x[+q]); `x` points at the centre, stride s
__device__ __forceinline__ float conv_even(const float* x, int s, const float* t, int K) {
    float acc = t[0] * x[0];
#pragma unroll
    for (int q = 1; q <= kMaxDerivRadius; ++q)
        if (q <= K) acc = fmaf(t[q], x[-q * s] + x[q * s], acc);
    return acc;
}

// odd taps under convolution: sum_q t[q] x[c - q] = sum_{q>0} t[q] (x[-q] - x[+q])
__device__ __forceinline__ float conv_odd(const float* x, int s, const float* t, int K) {
    float acc = 0.f;
#pragma unroll
    for (int q = 1; q <= kMaxDerivRadius; ++q)
        if (q <= K) acc = fmaf(t[q], x[-q * s] - x[q * s], acc);
    return acc;
}

// image samples to intensities: float as is; uint16 scaled to [0, 1] by
// v / 65535, correctly rounded: the product with the rounded reciprocal and one
// correction by its exact residual (Markstein's step), which gives the rounded
// quotient for each of the 65536 values (checked in exact arithmetic).  The
// division and the integer conversion (a quarter of the FP32 rate) took a third of
// the steering of a 16-bit image: 10000 x 10000, whole build 6342 -> 5704 us.
__device__ __forceinline__ float to_unit(float v) { return v; }
__device__ __forceinline__ float to_unit(uint16_t v) {
    constexpr float c = 1.f / 65535.f;
    const float x = __uint_as_float(0x4b000000u | v) - 8388608.f;
    const float q = __fmul_rn(x, c);
    return fmaf(fmaf(-q, 65535.f, x), c, q);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k_sfoc_steer(const T* __restrict__ img, int H, int W, size_t pitch,
                                                          float* __restrict__ F, size_t fpitch, size_t fplane,
                                                          SteerTaps tp) {
    extern __shared__ float sm[];
    const int hal = tp.halo;
    const int IW = kTW + 2 * hal, IH = kTH + 2 * hal;
    float* s_img = sm;
    float* s_h = s_img + IH * IW;
    const int plane = IH * kTW;
    const int x0 = blockIdx.x * kTW, y0 = blockIdx.y * kTH;

    for (int i = threadIdx.x; i < IH * IW; i += kThreads) {
        int r = i / IW, c = i - r * IW;
        int gy = clampi(y0 + r - hal, 0, H - 1), gx = clampi(x0 + c - hal, 0, W - 1);
        s_img[i] = to_unit(__ldg(img + (size_t)gy * pitch + gx));
    }
    __syncthreads();

    // horizontal passes.  planes: 2s = a1_s (odd), 2s+1 = g1_s (even);
    // second group: 2ns = a2 (even), 2ns+1 = g2 (even), 2ns+2 = c2x (odd)
    const int ns = tp.ns;
    for (int i = threadIdx.x; i < IH * kTW; i += kThreads) {
        int r = i / kTW, c = i - r * kTW;
        const float* x = s_img + r * IW + c + hal;
        for (int s = 0; s < ns; ++s) {
            s_h[(2 * s) * plane + i] = conv_odd(x, 1, tp.a1[s], tp.K1[s]);
            s_h[(2 * s + 1) * plane + i] = conv_even(x, 1, tp.g1[s], tp.K1[s]);
        }
        if (tp.second) {
            s_h[(2 * ns) * plane + i] = conv_even(x, 1, tp.a2, tp.K2);
            s_h[(2 * ns + 1) * plane + i] = conv_even(x, 1, tp.g2, tp.K2);
            s_h[(2 * ns + 2) * plane + i] = conv_odd(x, 1, tp.c2x, tp.K2);
        }
    }
    __syncthreads();

    for (int i = threadIdx.x; i < kTH * kTW; i += kThreads) {
        int r = i / kTW, c = i - r * kTW;
        int gy = y0 + r, gx = x0 + c;
        if (gy >= H || gx >= W) continue;
        const int off = (r + hal) * kTW + c;
        float Ix[kMaxScales], Iy[kMaxScales];
        for (int s = 0; s < ns; ++s) {
            Ix[s] = conv_even(s_h + (2 * s) * plane + off, kTW, tp.g1[s], tp.K1[s]);      // a1(x) g(y)
            Iy[s] = conv_odd(s_h + (2 * s + 1) * plane + off, kTW, tp.a1[s], tp.K1[s]);   // g(x) a1(y)
        }
        float* out = F + (size_t)gy * fpitch + gx;
        for (int k = 0; k < tp.no; ++k) {
            float f = 0.f;
            for (int s = 0; s < ns; ++s) {
                float v = fmaf(tp.ct[k], Ix[s], tp.st[k] * Iy[s]);
                f += tp.rectify ? fabsf(v) : v;
            }
            out[(size_t)k * fplane] = f;
        }
        if (tp.second) {
            float Ixx = conv_even(s_h + (2 * ns) * plane + off, kTW, tp.g2, tp.K2);      // a2(x) g2(y)
            float Iyy = conv_even(s_h + (2 * ns + 1) * plane + off, kTW, tp.a2, tp.K2);  // g2(x) a2(y)
            float Ixy = conv_odd(s_h + (2 * ns + 2) * plane + off, kTW, tp.c2y, tp.K2);  // c(x) c(y)
            for (int k = 0; k < tp.no; ++k) {
                float c2 = tp.ct[k] * tp.ct[k], s2 = tp.st[k] * tp.st[k], cs = 2.f * tp.st[k] * tp.ct[k];
                float v = fmaf(c2, Ixx, fmaf(s2, Iyy, -cs * Ixy));
                out[(size_t)(tp.no + k) * fplane] = tp.rectify ? fabsf(v) : v;
            }
        }
    }
}

// Steering at the paper's radii (three first-order scales of radii 2, 3, 3 and
// the second-order radius 5; six orientations).
//
// A warp takes a strip of 32 columns, a lane per column, and streams down its
// rows: from a row's window of 11 samples a lane makes the nine horizontal
// sums (sums and differences x[-q] +- x[q] shared by all nine) and adds each at
// once to the rows of its vertical pass, which are running sums in registers.
// Nothing but the image row passes through shared memory.  Rows are taken 4 at
// a time; first-order rows complete 3 rows behind the input, second-order rows
// 5, and are steered and written as they complete.
//
// What bounds it: writing the twelve planes (48 B per pixel), then ~180 FP32
// operations per pixel.  The tiled form this replaces (image tile with clamped
// element-wise loads, nine planes written to shared memory and read back)
// spent most of its time waiting for the tile.  2048 x 2048: 90 -> 53 us
// (the planes alone take 30).
constexpr int kSrW = 32, kSrU = 4, kSrThreads = 128, kSrPitch = 44;  // staged columns x0 - 5 .. x0 + 36

// output rows per warp of a batched launch (a single image's launch passes its own)
__host__ __device__ inline int steer_rows(int H) {
    const int seg = (H + 64) / 128 > 0 ? (H + 64) / 128 : 1;
    return ((H + seg - 1) / seg + kSrU - 1) / kSrU * kSrU;
}

// One or two images (`one`, warps = strips x segments in row-major order) or a batch
// (device table `jobs`, CTAs of image j from begin[j]).  seg_rows: output rows
// per warp (0: steer_rows of the image).
template <typename T>
__global__ void __launch_bounds__(kSrThreads, 3)
    k_sfoc_steer_strip(const __grid_constant__ ImgPair one, const ImgJob* __restrict__ jobs,
                       const int* __restrict__ begin, int n_jobs, const __grid_constant__ SteerTaps tp, int seg_rows) {
    constexpr int U = kSrU, N1 = U + 6, N2 = U + 10;
    __shared__ float s_rows[kSrThreads / 32][2][U][kSrPitch];
    int tile;
    const ImgJob& J = img_job(one, jobs, begin, n_jobs, &tile);
    const T* __restrict__ img = static_cast<const T*>(J.img);
    const int H = J.H, W = J.W;
    const size_t pitch = J.pitch, fpitch = J.fpitch, fplane = J.fpitch * (size_t)J.H;
    float* __restrict__ F = J.F;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int strips = (W + kSrW - 1) / kSrW;
    const int rows = seg_rows ? seg_rows : steer_rows(H);
    const int task = tile * (kSrThreads / 32) + warp;
    const int seg = task / strips;
    const int x0 = (task - seg * strips) * kSrW, y0 = seg * rows;
    if (y0 >= H) return;  // (no block barrier below)
    const int y1 = min(y0 + rows, H);
    const int gx = x0 + lane;
    const int xa = clampi(gx - 5, 0, W - 1), xb = clampi(gx + 27, 0, W - 1);  // this lane's staged columns

    float ix[3][N1], iy[3][N1], dxx[N2], dyy[N2], dxy[N2];
#pragma unroll
    for (int k = 0; k < N1; ++k)
#pragma unroll
        for (int q = 0; q < 3; ++q) ix[q][k] = iy[q][k] = 0.f;
#pragma unroll
    for (int k = 0; k < N2; ++k) dxx[k] = dyy[k] = dxy[k] = 0.f;

    float pa[U], pb[U];  // the next block's samples
    auto fetch = [&](int i0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const T* row = img + (size_t)clampi(i0 + u, 0, H - 1) * pitch;
            pa[u] = to_unit(__ldg(row + xa));
            pb[u] = lane < 10 ? to_unit(__ldg(row + xb)) : 0.f;
        }
    };
    fetch(y0 - 5);
    int buf = 0;
    for (int i0 = y0 - 5; i0 < y1 + 5; i0 += U, buf ^= 1) {
        float (*st)[kSrPitch] = s_rows[warp][buf];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            st[u][lane] = pa[u];
            if (lane < 10) st[u][32 + lane] = pb[u];
        }
        // one warp barrier a block: a buffer's readers are behind the next block's
        __syncwarp();
        if (i0 + U < y1 + 5) fetch(i0 + U);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float* x = &st[u][lane + 5];
            const float c = x[0];
            float e[6], o[6];
#pragma unroll
            for (int q = 1; q <= 5; ++q) {
                const float l = x[-q], r = x[q];
                e[q] = l + r;
                o[q] = l - r;
            }
            auto even = [&](const float* t, int K) {
                float v = t[0] * c;
#pragma unroll
                for (int q = 1; q <= 5; ++q)
                    if (q <= K) v = fmaf(t[q], e[q], v);
                return v;
            };
            auto odd = [&](const float* t, int K) {
                float v = t[1] * o[1];
#pragma unroll
                for (int q = 2; q <= 5; ++q)
                    if (q <= K) v = fmaf(t[q], o[q], v);
                return v;
            };
            // vertical: row i0 + u goes to rows i0 + u +- q; entry k of the first
            // order is row i0 + k - 3, of the second order row i0 + k - 5
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int K = q == 0 ? 2 : 3;
                const float ha = odd(tp.a1[q], K), hg = even(tp.g1[q], K);
                ix[q][u + 3] = fmaf(tp.g1[q][0], ha, ix[q][u + 3]);
#pragma unroll
                for (int d = 1; d <= 3; ++d)
                    if (d <= K) {
                        ix[q][u + 3 - d] = fmaf(tp.g1[q][d], ha, ix[q][u + 3 - d]);
                        ix[q][u + 3 + d] = fmaf(tp.g1[q][d], ha, ix[q][u + 3 + d]);
                        iy[q][u + 3 + d] = fmaf(tp.a1[q][d], hg, iy[q][u + 3 + d]);
                        iy[q][u + 3 - d] = fmaf(-tp.a1[q][d], hg, iy[q][u + 3 - d]);
                    }
            }
            const float hx = even(tp.a2, 5), hy = even(tp.g2, 5), hc = odd(tp.c2x, 5);
            dxx[u + 5] = fmaf(tp.g2[0], hx, dxx[u + 5]);
            dyy[u + 5] = fmaf(tp.a2[0], hy, dyy[u + 5]);
#pragma unroll
            for (int d = 1; d <= 5; ++d) {
                dxx[u + 5 - d] = fmaf(tp.g2[d], hx, dxx[u + 5 - d]);
                dxx[u + 5 + d] = fmaf(tp.g2[d], hx, dxx[u + 5 + d]);
                dyy[u + 5 - d] = fmaf(tp.a2[d], hy, dyy[u + 5 - d]);
                dyy[u + 5 + d] = fmaf(tp.a2[d], hy, dyy[u + 5 + d]);
                dxy[u + 5 + d] = fmaf(tp.c2y[d], hc, dxy[u + 5 + d]);
                dxy[u + 5 - d] = fmaf(-tp.c2y[d], hc, dxy[u + 5 - d]);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int ya = i0 + u - 3, yb = i0 + u - 5;
            if (gx < W && ya >= y0 && ya < y1) {
                float* out = F + (size_t)ya * fpitch + gx;
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    float f = 0.f;
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const float v = fmaf(tp.ct[k], ix[q][u], tp.st[k] * iy[q][u]);
                        f += tp.rectify ? fabsf(v) : v;
                    }
                    out[(size_t)k * fplane] = f;
                }
            }
            if (gx < W && yb >= y0 && yb < y1) {
                float* out = F + (size_t)yb * fpitch + gx;
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    const float c2 = tp.ct[k] * tp.ct[k], s2 = tp.st[k] * tp.st[k], cs = 2.f * tp.st[k] * tp.ct[k];
                    const float v = fmaf(c2, dxx[u], fmaf(s2, dyy[u], -cs * dxy[u]));
                    out[(size_t)(6 + k) * fplane] = tp.rectify ? fabsf(v) : v;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < N1; ++k)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                ix[q][k] = k + U < N1 ? ix[q][k + U] : 0.f;
                iy[q][k] = k + U < N1 ? iy[q][k + U] : 0.f;
            }
#pragma unroll
        for (int k = 0; k < N2; ++k) {
            dxx[k] = k + U < N2 ? dxx[k + U] : 0.f;
            dyy[k] = k + U < N2 ? dyy[k + U] : 0.f;
            dxy[k] = k + U < N2 ? dxy[k + U] : 0.f;
        }
    }
}

// Smoothing (Sec. 2.1): per channel, the F tile with the group's halo
// (clamped) is staged in shared memory; the horizontal pass of each rate
// runs register-blocked (a thread loads one row segment once and produces 8
// outputs for every rate) into shared planes; the vertical pass runs
// register-blocked too (8 rows of one column per thread) and sums the rates
// in registers.  The six channels of a group stay in registers, are
// normalised there and written out: F32 planar, or the bf16 chunks (chunk
// g = the six channels of group g and two zeros) in both pixel orders,
// plus the per-pixel sum planes.  Tiles are 32 columns x 64 rows.
constexpr int kSTW = 32, kSTH = 64, kSRows = 8;

template <int KD>
__device__ __forceinline__ void smooth_channel(const float* __restrict__ Fk, size_t fpitch, int H, int W, int x0,
                                               int y0, int hal, int n_dil, const int* s_dil, const float* t,
                                               float* s_F, int FW, float* s_h, int HR, float (&Dk)[kSRows]) {
    const int IW = kSTW + 2 * hal, IH = kSTH + 2 * hal;
    const int nd = KD > 0 ? n_dil : 1;  // radius 0: the group is unsmoothed, D = F (no sum over rates)
    __syncthreads();  // previous channel done with s_F / s_h
    // load: 8 threads per row, 8 consecutive columns each
    for (int rr = threadIdx.x >> 3; rr < IH; rr += kThreads >> 3) {
        const int yy = clampi(y0 + rr - hal, 0, H - 1);
        const float* row = Fk + (size_t)yy * fpitch;
        const int cb = (threadIdx.x & 7) * 8;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int cc = cb + c;
            if (cc < IW) s_F[rr * FW + cc] = __ldg(row + clampi(x0 + cc - hal, 0, W - 1));
        }
    }
    __syncthreads();
    // horizontal: task = (row, 8-column block); 4 blocks per row
    for (int task = threadIdx.x; task < IH * 4; task += kThreads) {
        const int rr = task >> 2, cb = (task & 3) * 8;
        const float* x = s_F + rr * FW + cb;  // x[c + hal] is column cb + c
        for (int ri = 0; ri < nd; ++ri) {
            const int rate = s_dil[ri];
            float o[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) o[c] = t[0] * x[c + hal];
#pragma unroll
            for (int q = 1; q <= KD; ++q) {
                const float tq = t[q];
#pragma unroll
                for (int c = 0; c < 8; ++c) o[c] = fmaf(tq, x[c + hal - q * rate] + x[c + hal + q * rate], o[c]);
            }
            float4* dst = reinterpret_cast<float4*>(s_h + (ri * HR + rr) * kSTW + cb);
            dst[0] = make_float4(o[0], o[1], o[2], o[3]);
            dst[1] = make_float4(o[4], o[5], o[6], o[7]);
        }
    }
    __syncthreads();
    // vertical: task = (column, 8-row block): 32 x 8 = 256 tasks
    const int col = threadIdx.x & 31, rb = (threadIdx.x >> 5) * kSRows;
#pragma unroll
    for (int j = 0; j < kSRows; ++j) Dk[j] = 0.f;
    for (int ri = 0; ri < nd; ++ri) {
        const int rate = s_dil[ri];
        const float* x = s_h + (ri * HR + rb + hal) * kSTW + col;  // x[j * kSTW] is output row rb + j
#pragma unroll
        for (int j = 0; j < kSRows; ++j) {
            float a = t[0] * x[j * kSTW];
#pragma unroll
            for (int q = 1; q <= KD; ++q) a = fmaf(t[q], x[(j - q * rate) * kSTW] + x[(j + q * rate) * kSTW], a);
            Dk[j] += a;
        }
    }
}

// Normalises one pixel's group of `no` smoothed values d[k] (Sec. 2.1) and
// writes it out: F32 planes, or the bf16 chunk in both pixel orders and the
// bf16 planes; adds
// the stored values to the per-pixel sums a1 (g) and a2 (g^2).
template <int NO, int KO>
__device__ __forceinline__ void write_pixel(int g, int no, const float* d, float eps, int gy, int gx, int H, int W,
                                            float* __restrict__ c32, size_t cpitch, size_t cplane,
                                            __nv_bfloat16* __restrict__ rm, __nv_bfloat16* __restrict__ cm,
                                            __nv_bfloat16* __restrict__ pl, float& a1, float& a2) {
    const bool bf = rm != nullptr;
    float n2 = 0.f;
#pragma unroll
    for (int k = 0; k < KO; ++k)
        if (k < no) n2 = fmaf(d[k], d[k], n2);
    const float den = sqrtf(n2) + eps;
    const float inv = den > 0.f ? 1.f / den : 0.f;  // NaN stays NaN through d * inv
    const bool in = gy < H && gx < W;
    float vs[KO];
#pragma unroll
    for (int k = 0; k < KO; ++k) {
        if (k >= no) break;
        float v = (den > 0.f || den != den) ? d[k] * inv : 0.f;
        if (bf) v = __bfloat162float(__float2bfloat16_rn(v));
        vs[k] = v;
        a1 += v;
        a2 = fmaf(v, v, a2);
        if (c32 && in) c32[(size_t)(g * no + k) * cplane + (size_t)gy * cpitch + gx] = v;
    }
    if constexpr (NO == 6) {
        if (bf && in) {  // chunk g: the six channels, then two zeros
            auto pack = [](float lo, float hi) {
                const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
                return *reinterpret_cast<const unsigned*>(&h);
            };
            const uint4 chunk = make_uint4(pack(vs[0], vs[1]), pack(vs[2], vs[3]), pack(vs[4], vs[5]), 0u);
            const size_t npx = (size_t)H * W;
            const size_t pix = (size_t)gy * W + gx, cpx = (size_t)gx * H + gy;
            *reinterpret_cast<uint4*>(rm + ((size_t)g * npx + pix) * 8) = chunk;
            *reinterpret_cast<uint4*>(cm + ((size_t)g * npx + cpx) * 8) = chunk;
            // the planes, from the chunk's halves (a conversion per channel of their own
            // and 64-bit addresses made these builds 3 to 5 % slower)
            unsigned short* q = reinterpret_cast<unsigned short*>(pl) + (size_t)g * 6 * cplane + (size_t)gy * cpitch + gx;
            const unsigned h[3] = {chunk.x, chunk.y, chunk.z};
#pragma unroll
            for (int k = 0; k < 6; ++k, q += cplane) *q = (unsigned short)(h[k >> 1] >> (16 * (k & 1)));
        }
    }
}

// One group of `no` channels with radius and rates at run time: smooth each
// channel, normalise the group in registers and write it out.
template <int NO>
__device__ __forceinline__ void smooth_group(int g, const float* __restrict__ F, size_t fpitch, size_t fplane, int H,
                                             int W, const SmoothTaps& tp, const int* s_dil, const float* t,
                                             float* s_F, int FW, float* s_h, int HR, int x0,
                                             int y0, float* __restrict__ c32, size_t cpitch, size_t cplane,
                                             __nv_bfloat16* __restrict__ rm, __nv_bfloat16* __restrict__ cm,
                                             __nv_bfloat16* __restrict__ pl,
                                             float (&a1)[kSRows], float (&a2)[kSRows]) {
    constexpr int KO = NO > 0 ? NO : kMaxOrient;
    const int no = NO > 0 ? NO : tp.no;
    const int col = threadIdx.x & 31, rb = (threadIdx.x >> 5) * kSRows;
    const int gx = x0 + col;
    float D[KO][kSRows];
#pragma unroll
    for (int k = 0; k < KO; ++k) {
        if (k >= no) break;
        const float* Fk = F + (size_t)(g * no + k) * fplane;
        {
            const int hal = tp.halo[g], Kd = tp.Kd[g];
            switch (Kd) {
                case 0: smooth_channel<0>(Fk, fpitch, H, W, x0, y0, hal, tp.n_dil, s_dil, t, s_F, FW, s_h, HR, D[k]); break;
                case 1: smooth_channel<1>(Fk, fpitch, H, W, x0, y0, hal, tp.n_dil, s_dil, t, s_F, FW, s_h, HR, D[k]); break;
                case 2: smooth_channel<2>(Fk, fpitch, H, W, x0, y0, hal, tp.n_dil, s_dil, t, s_F, FW, s_h, HR, D[k]); break;
                case 3: smooth_channel<3>(Fk, fpitch, H, W, x0, y0, hal, tp.n_dil, s_dil, t, s_F, FW, s_h, HR, D[k]); break;
                case 4: smooth_channel<4>(Fk, fpitch, H, W, x0, y0, hal, tp.n_dil, s_dil, t, s_F, FW, s_h, HR, D[k]); break;
                case 5: smooth_channel<5>(Fk, fpitch, H, W, x0, y0, hal, tp.n_dil, s_dil, t, s_F, FW, s_h, HR, D[k]); break;
                default: smooth_channel<6>(Fk, fpitch, H, W, x0, y0, hal, tp.n_dil, s_dil, t, s_F, FW, s_h, HR, D[k]); break;
            }
        }
    }
    // group normalisation in registers; write this group
#pragma unroll
    for (int j = 0; j < kSRows; ++j) {
        float d[KO];
#pragma unroll
        for (int k = 0; k < KO; ++k) d[k] = D[k][j];
        write_pixel<NO, KO>(g, no, d, tp.eps, y0 + rb + j, gx, H, W, c32, cpitch, cplane, rm, cm, pl, a1[j], a2[j]);
    }
}

// The paper's dilation rates 1, 2, 3 with smoothing radius KD at compile time,
// one group g per launch (the second group's launch continues the per-pixel
// sums from the stored planes, adding in the same order as one launch would).
//
// A CTA takes a strip of 64 columns and streams down its rows, one warp per
// channel of the group, a lane per column pair.  A lane takes its window of an
// input row from shared memory once (LDS.64 pairs), makes the row's three
// horizontal sums in registers and adds them at once to the output rows they
// belong to: rate r, tap q of row i goes to row i + q r, so the vertical pass
// is 2 hal + 8 running sums per column in registers and touches no shared
// memory.  Rows are taken 8 at a time; the 8 rows a block completes go to
// shared memory, where two more warps meet the group's six channels of a pixel,
// normalise and write them, while the channel warps are on the next block
// (named barriers hand the two buffers over; with the channel warps doing this
// themselves behind block barriers the kernel was 1.5x slower).
//
// What bounds it: per pixel and channel the 2 x 3 (2 KD + 1) multiply-adds
// take 66 / 128 clocks of an SM at KD = 5, and the window reads 34 / 64.  The
// tiled form this replaces (horizontal sums of every rate written to shared
// memory, read back by the vertical pass, 32 x 64 tiles that redo 1.5x of the
// horizontal work) needed 30 shared words and ~90 instructions per pixel and
// channel against 17 and ~50 here, with block barriers between its passes.
// The finishing warps are as busy as the channel warps: without a branch per
// column in them both groups of 1847 x 2891 took 330 us instead of 449.
// Both groups of a 2048 x 2048 image: 322 -> 207 us (F32 cube), 343 -> 226 (BF16).
constexpr int kStW = 64;     // strip width: 32 lanes x 2 columns
constexpr int kStU = 8;      // rows per block
constexpr int kStH = 4;      // rows between two shifts of the running sums
constexpr int kStChan = 6, kStFin = 2;  // channel warps, finishing warps
constexpr int kStThreads = (kStChan + kStFin) * 32;

template <int KD>
struct StripGeom {
    static constexpr int HAL = 3 * KD;
    static constexpr int OFF = (HAL + 3) / 4 * 4;             // shared column of the strip's first column
    static constexpr int RW = (OFF + kStW + HAL + 1 + 3) / 4 * 4;  // floats per staged row
    static constexpr int NW2 = HAL + 2;                        // window, float2
    static constexpr int NA = 2 * HAL + kStH;                  // running sums
    static constexpr int LEAD = (2 * HAL + kStU - 1) / kStU;   // blocks before the first completed rows
    // per CTA: staged rows (two blocks per channel), completed rows and bf16
    // chunks (two blocks each)
    static constexpr size_t rows_f = (size_t)6 * 2 * kStU * RW;
    static constexpr size_t done_f = (size_t)2 * 6 * kStU * kStW;
    static constexpr int CP = kStW + 1;                        // chunk row pitch (16-byte units)
    static constexpr size_t smem = sizeof(float) * (rows_f + done_f) + 16 * (size_t)2 * kStU * CP;
};

// output rows per CTA of a batched launch (a single image's launch passes its own)
__host__ __device__ inline int strip_rows(int H) {
    const int seg = (H + 128) / 256 > 0 ? (H + 128) / 256 : 1;
    return ((H + seg - 1) / seg + kStU - 1) / kStU * kStU;
}

// Copies kStU rows of one channel from row i0 (clamped to the image) into dst;
// one commit group.  Pieces of 16 bytes inside the rows (rows and x0 - OFF are
// 16-byte aligned), and on the image's left and right strips the clamped columns
// one by one, 16 of a row at a time.  (Copying such a strip's rows element by
// element made its CTAs issue 1.4 times the instructions of the others, and a
// launch of one wave waited for them: 512 x 512 19.4 and 25.9 us for groups 0 and
// 1, with this 17.5 and 23.6.  A right strip of few columns was worse still, until
// it left out the columns past the halo: both groups of 1847 x 2891, 11 columns in
// the last strip, 562 -> 449 us.)
template <int KD>
__device__ __forceinline__ void strip_rows_async(const float* __restrict__ Fk, size_t fpitch, int H, int W, int x0,
                                                 int i0, float* dst, int lane) {
    using G = StripGeom<KD>;
    static_assert(G::OFF <= 16 && G::RW / 4 <= 32, "a lane per piece, one step left of the image");
    const int xs = x0 - G::OFF;
    const int xl = xs + 4 * lane;
    const bool whole = lane < G::RW / 4 && xl >= 0 && xl + 4 <= W;
#pragma unroll
    for (int u = 0; u < kStU; ++u) {
        const float* src = Fk + (size_t)clampi(i0 + u, 0, H - 1) * fpitch + xl;
        const unsigned d = (unsigned)__cvta_generic_to_shared(dst + u * G::RW + 4 * lane);
        if (whole) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    }
    auto clamped = [&](int c0, int c1) {  // columns [c0, min(c0 + 16, c1)) of the staged rows
        const int c = c0 + (lane & 15);
        const float* col = Fk + clampi(xs + c, 0, W - 1);
        if (c < c1)
#pragma unroll
            for (int u = lane >> 4; u < kStU; u += 2) {
                const unsigned d = (unsigned)__cvta_generic_to_shared(dst + u * G::RW + c);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d),
                             "l"(col + (size_t)clampi(i0 + u, 0, H - 1) * fpitch)
                             : "memory");
            }
    };
    if (xs < 0) clamped(0, -xs);
    // (W > x0, so the first piece that is not whole is right of those.)  Columns past
    // W - 1 + HAL reach no column of the image: they stay as they are
    const int cend = W + G::HAL - xs < G::RW ? W + G::HAL - xs : G::RW;
    for (int c0 = (W & ~3) - xs; c0 < cend; c0 += 16) clamped(c0, cend);
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The column-order bf16 chunks of a completed block: 8 lanes take the 8 rows of
// one column, so that a column's 128 contiguous bytes leave together; a thread
// keeps its row and steps over every eighth column.  tid: 0 .. 32 kStFin - 1.
__device__ __forceinline__ void strip_write_cm(const ImgJob& J, int g, const uint4* s_chunk, int cp, int x0, int yb,
                                               int y1, int tid) {
    constexpr int kStep = kStFin * 32 / kStU;
    const int c0 = tid / kStU, u = tid % kStU;
    if (yb + u >= y1) return;
    uint4* q = reinterpret_cast<uint4*>(J.cm) + ((size_t)g * J.W + x0 + c0) * J.H + yb + u;
    const size_t step = (size_t)kStep * J.H;
    const uint4* src = s_chunk + u * cp + c0;
#pragma unroll
    for (int c = 0; c < kStW; c += kStep, q += step)
        if (x0 + c0 + c < J.W) *q = src[c];
}

// Where a finishing warp's lane writes: its two pixels of row 0, and what holds
// for every row.
struct StripOut {
    float* s1;
    float* s2;
    float* c32;   // group g's first plane (or nullptr)
    uint4* rm;    // group g's chunks (or nullptr)
    __nv_bfloat16* pl;  // group g's first bf16 plane (with rm)
    size_t pitch, plane;
    int W;
    bool two;     // the second pixel is inside the image
    bool vec;     // planes take both columns in one store: the pitch is even, so that the second one is inside the
                  // row's padding at worst, and every row starts on 8 bytes.  (A lane of an odd width that stored
                  // one column made its strip's warps run both forms: 1 / 6 of the time.)  A dense cube of odd
                  // width (sfoc_build_static) is not
};

// One completed row of a strip: a lane normalises its two pixels' six channels
// (as write_pixel does) and writes the F32 planes, or the bf16 chunks, and the
// per-pixel sums, continued from `sums` (g of both pixels, then g^2).
// `done`: the row's [channel][8][64] values at the lane's columns; `chunk`: the
// lane's place in the chunk buffer.
template <bool VEC>
__device__ __forceinline__ void strip_finish(const StripOut& o, float eps, const float* done, uint4* chunk, int gy,
                                             const float4& sums) {
    float2 d[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) d[k] = *reinterpret_cast<const float2*>(done + k * kStU * kStW);
    float a1[2] = {sums.x, sums.y}, a2[2] = {sums.z, sums.w};
    const bool bf = o.rm != nullptr;
    float v[2][6];
    unsigned pk[2][3];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        float n2 = 0.f;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const float x = e ? d[k].y : d[k].x;
            n2 = fmaf(x, x, n2);
        }
        const float den = sqrtf(n2) + eps;
        const float inv = den > 0.f ? 1.f / den : 0.f;  // NaN stays NaN through d * inv, and 0 / 0 is 0
#pragma unroll
        for (int k = 0; k < 6; ++k) v[e][k] = (e ? d[k].y : d[k].x) * inv;
        if (bf) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const __nv_bfloat162 h = __floats2bfloat162_rn(v[e][2 * k], v[e][2 * k + 1]);
                pk[e][k] = *reinterpret_cast<const unsigned*>(&h);
                v[e][2 * k] = __uint_as_float(pk[e][k] << 16);
                v[e][2 * k + 1] = __uint_as_float(pk[e][k] & 0xffff0000u);
            }
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            a1[e] += v[e][k];
            a2[e] = fmaf(v[e][k], v[e][k], a2[e]);
        }
    }
    const size_t at = (size_t)gy * o.pitch;
    auto put2 = [&](float* q, float x, float y) {
        if (VEC) {
            *reinterpret_cast<float2*>(q) = make_float2(x, y);
        } else {
            q[0] = x;
            if (o.two) q[1] = y;
        }
    };
    put2(o.s1 + at, a1[0], a1[1]);
    put2(o.s2 + at, a2[0], a2[1]);
    if (o.c32) {
        float* q = o.c32 + at;
#pragma unroll
        for (int k = 0; k < 6; ++k, q += o.plane) put2(q, v[0][k], v[1][k]);
    }
    if (bf) {
        __nv_bfloat16* q = o.pl + at;  // (BF16 cubes are padded: both columns in one store)
#pragma unroll
        for (int k = 0; k < 6; ++k, q += o.plane)
            *reinterpret_cast<unsigned*>(q) = __byte_perm(pk[0][k >> 1], pk[1][k >> 1], (k & 1) ? 0x7632 : 0x5410);
        uint4* const rm = o.rm + (size_t)gy * o.W;
#pragma unroll
        for (int e = 0; e < 2; ++e) {  // chunk g: the six channels, then two zeros
            const uint4 c = make_uint4(pk[e][0], pk[e][1], pk[e][2], 0u);
            if (e == 0 || o.two) rm[e] = c;
            chunk[e] = c;
        }
    }
}

// One or two images (`one`, CTA = strip of the image's strips x segments) or a batch
// (device table `jobs`, CTAs of image j from begin[j]).  seg_rows: output rows
// per CTA, a multiple of kStU (0: strip_rows of the image).
template <int KD>
__global__ void __launch_bounds__(kStThreads, 2)
    k_sfoc_smooth_strip(const __grid_constant__ ImgPair one, const ImgJob* __restrict__ jobs,
                        const int* __restrict__ begin, int n_jobs, const __grid_constant__ SmoothTaps tp, int g,
                        int seg_rows) {
    using G = StripGeom<KD>;
    constexpr int HAL = G::HAL, U = kStU, UH = kStH;
    constexpr int kFull = 1, kEmpty = 3, kPair = 5;  // named barriers (two buffers each; the finishing warps' own)
    extern __shared__ __align__(16) float sm[];
    float* s_rows = sm;                 // [channel][2][U][RW]
    float* s_done = s_rows + G::rows_f;  // [2][channel][U][kStW]
    uint4* s_chunk = reinterpret_cast<uint4*>(s_done + G::done_f);  // [2][U][CP]
    int tile;
    const ImgJob& J = img_job(one, jobs, begin, n_jobs, &tile);
    const int H = J.H, W = J.W;
    const int strips = (W + kStW - 1) / kStW;
    const int rows = seg_rows ? seg_rows : strip_rows(H);
    const int seg = tile / strips;
    const int x0 = (tile - seg * strips) * kStW, y0 = seg * rows;
    const int y1 = min(y0 + rows, H);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nout = (y1 - y0 + U - 1) / U;  // blocks of completed rows
    // the first group's launch lets the second one's start beside it; the second
    // one reads only F (complete before the first began) until its finishing warps
    // have waited for the first to end
    if (g == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (warp >= kStChan) {
        if (g) asm volatile("griddepcontrol.wait;" ::: "memory");
        // ---- finishing warps: rows warp - kStChan, + kStFin, ... of each block
        const int gx = x0 + 2 * lane;
        const size_t plane = J.cpitch * (size_t)H;
        StripOut o;
        o.s1 = J.s1 + gx;
        o.s2 = J.s2 + gx;
        o.c32 = J.c32 ? J.c32 + (size_t)g * 6 * plane + gx : nullptr;
        o.rm = J.rm ? reinterpret_cast<uint4*>(J.rm) + (size_t)g * H * W + gx : nullptr;
        o.pl = J.pl ? J.pl + (size_t)g * 6 * plane + gx : nullptr;
        o.pitch = J.cpitch;
        o.plane = plane;
        o.W = W;
        o.two = gx + 1 < W;
        o.vec = (J.cpitch & 1) == 0 && ((reinterpret_cast<uintptr_t>(J.s1) | reinterpret_cast<uintptr_t>(J.s2) |
                                         reinterpret_cast<uintptr_t>(J.c32)) & 7) == 0;
        for (int m = 0; m < nout; ++m) {
            const int b = m & 1, yb = y0 + m * U + warp - kStChan;
            float4 sums[U / kStFin];
#pragma unroll
            for (int v = 0; v < U / kStFin; ++v) {
                const int gy = yb + v * kStFin;
                sums[v] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (g > 0 && gy < y1 && gx < W) {
                    const size_t at = (size_t)gy * o.pitch;
                    if (o.vec) {
                        const float2 a = *reinterpret_cast<const float2*>(o.s1 + at);
                        const float2 b = *reinterpret_cast<const float2*>(o.s2 + at);
                        sums[v] = make_float4(a.x, a.y, b.x, b.y);
                    } else {
                        sums[v].x = o.s1[at];
                        sums[v].z = o.s2[at];
                        if (o.two) {
                            sums[v].y = o.s1[at + 1];
                            sums[v].w = o.s2[at + 1];
                        }
                    }
                }
            }
            __syncwarp();
            asm volatile("bar.sync %0, %1;" ::"r"(kFull + b), "n"(kStThreads) : "memory");
            const float* done = s_done + (size_t)b * kStChan * U * kStW + (warp - kStChan) * kStW + 2 * lane;
            uint4* chunk = s_chunk + (size_t)b * U * G::CP + (warp - kStChan) * G::CP + 2 * lane;
            auto finish = [&](auto vec) {
#pragma unroll
                for (int v = 0; v < U / kStFin; ++v)
                    if (yb + v * kStFin < y1 && gx < W)
                        strip_finish<decltype(vec)::value>(o, tp.eps, done + v * kStFin * kStW,
                                                           chunk + v * kStFin * G::CP, yb + v * kStFin, sums[v]);
            };
            if (o.vec) finish(std::true_type());
            else finish(std::false_type());
            __syncwarp();
            if (m + 2 < nout) asm volatile("bar.arrive %0, %1;" ::"r"(kEmpty + b), "n"(kStThreads) : "memory");
            if (J.cm) {  // (a chunk buffer's next writer is behind the next block's barrier)
                asm volatile("bar.sync %0, %1;" ::"r"(kPair), "n"(kStFin * 32) : "memory");
                strip_write_cm(J, g, s_chunk + (size_t)b * U * G::CP, G::CP, x0, y0 + m * U, y1,
                               (int)threadIdx.x - kStChan * 32);
                __syncwarp();
            }
        }
        return;
    }
    // ---- channel warps
    const size_t fpitch = J.fpitch, fplane = J.fpitch * (size_t)J.H;
    const float* __restrict__ Fk = J.F + (size_t)(g * kStChan + warp) * fplane;
    float* const ring = s_rows + (size_t)warp * 2 * U * G::RW;
    float2 tq[KD + 1];
#pragma unroll
    for (int q = 0; q <= KD; ++q) {
        const float t = g ? tp.g[1][q] : tp.g[0][q];
        tq[q] = make_float2(t, t);
    }
    float2 a[G::NA];  // a[k]: output row i0 + k - HAL of the rows that start at input row i0
#pragma unroll
    for (int k = 0; k < G::NA; ++k) a[k] = make_float2(0.f, 0.f);

    // input rows from i0 = y0 - (LEAD U - HAL), so that block LEAD completes y0 .. y0 + U - 1
    const int first = y0 + HAL - G::LEAD * U;
    const int nb = G::LEAD + nout;
    strip_rows_async<KD>(Fk, fpitch, H, W, x0, first, ring, lane);
#pragma unroll 1
    for (int n = 0; n < nb; ++n) {
        if (n + 1 < nb) {
            strip_rows_async<KD>(Fk, fpitch, H, W, x0, first + (n + 1) * U, ring + ((n + 1) & 1) * U * G::RW, lane);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncwarp();  // every lane's copies of the block have landed
        const int m = n - G::LEAD;
        float* done = s_done + (size_t)((m & 1) * kStChan + warp) * U * kStW + 2 * lane;
        if (m >= 2) asm volatile("bar.sync %0, %1;" ::"r"(kEmpty + (m & 1)), "n"(kStThreads) : "memory");
        const float* blk = ring + (n & 1) * U * G::RW + (G::OFF - HAL - 1) + 2 * lane;
#pragma unroll 1
        for (int uh = 0; uh < U; uh += UH) {
#pragma unroll
            for (int u = 0; u < UH; ++u) {
                float2 w[G::NW2];  // shared columns OFF + 2 lane - HAL - 1 ...
#pragma unroll
                for (int v = 0; v < G::NW2; ++v) w[v] = *reinterpret_cast<const float2*>(blk + u * G::RW + 2 * v);
#pragma unroll
                for (int r = 1; r <= 3; ++r) {
                    // horizontal sum of rate r at both columns, outer taps first
                    float2 h = make_float2(0.f, 0.f);
#pragma unroll
                    for (int q = KD; q >= 1; --q) {
#pragma unroll
                        for (int sg = -1; sg <= 1; sg += 2) {
                            const int s = HAL + 1 + sg * q * r;  // window index of column 0's sample
                            const bool firstt = q == KD && sg < 0;
                            if (s % 2 == 0) {
                                h = firstt ? __fmul2_rn(tq[q], w[s / 2]) : __ffma2_rn(tq[q], w[s / 2], h);
                            } else {
                                h.x = firstt ? tq[q].x * w[s / 2].y : fmaf(tq[q].x, w[s / 2].y, h.x);
                                h.y = firstt ? tq[q].x * w[s / 2 + 1].x : fmaf(tq[q].x, w[s / 2 + 1].x, h.y);
                            }
                        }
                    }
                    h = __ffma2_rn(tq[0], w[(HAL + 1) / 2], h);
                    // row i = i0 + u of rate r belongs to output rows i + q r
#pragma unroll
                    for (int q = -KD; q <= KD; ++q)
                        a[u + HAL + q * r] = __ffma2_rn(tq[q < 0 ? -q : q], h, a[u + HAL + q * r]);
                }
            }
            blk += UH * G::RW;
            if (m >= 0) {
#pragma unroll
                for (int u = 0; u < UH; ++u) *reinterpret_cast<float2*>(done + (uh + u) * kStW) = a[u];
            }
#pragma unroll
            for (int k = 0; k < G::NA; ++k) a[k] = k + UH < G::NA ? a[k + UH] : make_float2(0.f, 0.f);
        }
        __syncwarp();  // the block's rows are read before the copies of block n + 2 replace them
        if (m >= 0) asm volatile("bar.arrive %0, %1;" ::"r"(kFull + (m & 1)), "n"(kStThreads) : "memory");
    }
}

// Any radii and rates at run time.
template <int NO>
__global__ void __launch_bounds__(kThreads, 1)
    k_sfoc_smooth(const float* __restrict__ F, size_t fpitch, size_t fplane, int H, int W, SmoothTaps tp,
                  float* __restrict__ c32, size_t cpitch, size_t cplane, __nv_bfloat16* __restrict__ rm,
                  __nv_bfloat16* __restrict__ cm, __nv_bfloat16* __restrict__ pl, float* __restrict__ s1,
                  float* __restrict__ s2) {
    extern __shared__ float sm[];
    __shared__ float s_tap[2][kMaxSmoothRadius + 1];  // taps in shared memory: no local copy of the params
    __shared__ int s_dil[kMaxDil];
    if (threadIdx.x < 2 * (kMaxSmoothRadius + 1)) {
        const int gg = threadIdx.x / (kMaxSmoothRadius + 1), q = threadIdx.x % (kMaxSmoothRadius + 1);
        s_tap[gg][q] = tp.g[gg][q];
    }
    if (threadIdx.x < kMaxDil) s_dil[threadIdx.x] = tp.dil[threadIdx.x];
    const int maxhal = max(tp.halo[0], tp.halo[1]);
    const int FW = smooth_row_stride(maxhal);
    const int HR = kSTH + 2 * maxhal;
    float* s_F = sm;             // HR x FW
    float* s_h = s_F + HR * FW;  // n_dil x HR x kSTW
    const int x0 = blockIdx.x * kSTW, y0 = blockIdx.y * kSTH;
    const int col = threadIdx.x & 31, rb = (threadIdx.x >> 5) * kSRows;
    const int gx = x0 + col;
    const int no = NO > 0 ? NO : tp.no;
    const int ng = tp.z / no;

    float a1[kSRows], a2[kSRows];
#pragma unroll
    for (int j = 0; j < kSRows; ++j) a1[j] = a2[j] = 0.f;
    for (int g = 0; g < ng; ++g)
        smooth_group<NO>(g, F, fpitch, fplane, H, W, tp, s_dil, s_tap[g], s_F, FW, s_h, HR, x0, y0, c32, cpitch,
                         cplane, rm, cm, pl, a1, a2);
#pragma unroll
    for (int j = 0; j < kSRows; ++j) {
        const int gy = y0 + rb + j;
        if (gy < H && gx < W) {
            s1[(size_t)gy * cpitch + gx] = a1[j];
            s2[(size_t)gy * cpitch + gx] = a2[j];
        }
    }
}

bool smooth_is_paper(const SmoothTaps& tp) {
    return tp.no == 6 && tp.z == 12 && tp.n_dil == 3 && tp.dil[0] == 1 && tp.dil[1] == 2 && tp.dil[2] == 3 &&
           tp.Kd[0] == 3 && tp.Kd[1] == 5;
}

__global__ void k_cube_export_bf16(const __nv_bfloat16* __restrict__ rm, int H, int W, int z, float* __restrict__ out) {
    size_t n = (size_t)H * W;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n * z; i += (size_t)gridDim.x * blockDim.x) {
        int k = (int)(i / n);
        size_t p = i - (size_t)k * n;
        int chunk = k / 6, j = k % 6;  // chunk g = the six channels of group g + two zeros
        out[i] = __bfloat162float(rm[((size_t)chunk * n + p) * 8 + j]);
    }
}

__global__ void k_cube_export_f32(const float* __restrict__ c32, int H, int W, int z, size_t pitch, float* __restrict__ out) {
    size_t n = (size_t)H * W;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n * z; i += (size_t)gridDim.x * blockDim.x) {
        int k = (int)(i / n);
        size_t p = i - (size_t)k * n;
        int y = (int)(p / W), x = (int)(p - (size_t)y * W);
        out[i] = c32[((size_t)k * H + y) * pitch + x];
    }
}

bool steer_is_paper(const SteerTaps& tp) {
    return tp.ns == 3 && tp.K1[0] == 2 && tp.K1[1] == 3 && tp.K1[2] == 3 && tp.second && tp.K2 == 5 && tp.no == 6;
}

int steer_ctas(int H, int W, int rows) {
    const int tasks = ((W + kSrW - 1) / kSrW) * ((H + rows - 1) / rows);
    return (tasks + kSrThreads / 32 - 1) / (kSrThreads / 32);
}

ImgPair img_none() {
    ImgPair p;
    memset(&p, 0, sizeof(p));
    p.split = 0x7fffffff;
    return p;
}

// Output rows per warp for one or two images: the rows with the least waves
// (three CTAs of four warps per SM) x rows streamed (10 more than the output
// rows).
int steer_rows_for(const ImgJob* j, int n) {
    const int slots = 3 * device_sms();
    int H = 0;
    for (int i = 0; i < n; ++i) H = j[i].H > H ? j[i].H : H;
    long best = -1;
    int rows = kSrU;
    for (int r = 4 * kSrU; r < H + kSrU; r += kSrU) {
        long ctas = 0;
        for (int i = 0; i < n; ++i) ctas += steer_ctas(j[i].H, j[i].W, r);
        const long cost = (ctas + slots - 1) / slots * (r + 14);
        if (best < 0 || cost <= best) {
            best = cost;
            rows = r;
        }
        if (ctas <= slots / 2) break;  // one partial wave already: longer segments only take longer
    }
    return rows;
}

template <typename T>
cudaError_t launch_steer_any(const T* img, int H, int W, size_t pitch, float* F, size_t fpitch, const SteerTaps& tp,
                             cudaStream_t st) {
    dim3 grid((W + kTW - 1) / kTW, (H + kTH - 1) / kTH);
    // the paper's scales (0.6, 0.8, 1.0 and 1.5 at 3 sigma: radii 2, 3, 3, 5), six orientations
    if (steer_is_paper(tp)) {
        ImgPair one = img_none();
        one.j[0].img = img;
        one.j[0].pitch = pitch;
        one.j[0].H = H;
        one.j[0].W = W;
        one.j[0].F = F;
        one.j[0].fpitch = fpitch;
        const int rows = steer_rows_for(&one.j[0], 1);
        k_sfoc_steer_strip<T><<<steer_ctas(H, W, rows), kSrThreads, 0, st>>>(one, nullptr, nullptr, 0, tp, rows);
        return cudaGetLastError();
    }
    const int hal = tp.halo;
    const int IH = kTH + 2 * hal, IW = kTW + 2 * hal;
    const int np = 2 * tp.ns + (tp.second ? 3 : 0);
    size_t smem = sizeof(float) * ((size_t)IH * IW + (size_t)np * IH * kTW);
    cudaError_t e = cudaFuncSetAttribute(k_sfoc_steer<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_sfoc_steer<T><<<grid, kThreads, smem, st>>>(img, H, W, pitch, F, fpitch, fpitch * (size_t)H, tp);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sfoc_steer(const float* img, int H, int W, size_t pitch, float* F, size_t fpitch,
                              const SteerTaps& tp, cudaStream_t st) {
    return launch_steer_any(img, H, W, pitch, F, fpitch, tp, st);
}

cudaError_t launch_sfoc_steer(const uint16_t* img, int H, int W, size_t pitch, float* F, size_t fpitch,
                              const SteerTaps& tp, cudaStream_t st) {
    return launch_steer_any(img, H, W, pitch, F, fpitch, tp, st);
}

int smooth_launch_count(const SmoothTaps& tp) { return smooth_is_paper(tp) ? 2 : 1; }

namespace {

// the two group launches of the paper's smoothing (sigma_d 1.0 / 1.5, rates
// 1, 2, 3) over `ctas` CTAs of seg_rows output rows (0: a batch's own)
cudaError_t launch_smooth_paper(const ImgPair& one, const ImgJob* jobs, const int* begin, int n_jobs, int ctas,
                                int seg_rows, const SmoothTaps& tp, cudaStream_t st) {
    auto run = [&](auto kern, int g, size_t smem) -> cudaError_t {
        const cudaError_t e2 = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e2 != cudaSuccess) return e2;
        // The second group may start while the first one's last CTAs run (it needs
        // of them only the sum planes, which its finishing warps wait for): the
        // first launch's partial last wave, or the half-empty chip of a small
        // image, does not idle.
        cudaLaunchAttribute early;
        early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        early.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3((unsigned)ctas);
        cfg.blockDim = dim3(kStThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cfg.attrs = &early;
        cfg.numAttrs = g ? 1 : 0;
        return cudaLaunchKernelEx(&cfg, kern, one, jobs, begin, n_jobs, tp, g, seg_rows);
    };
    cudaError_t e = run(k_sfoc_smooth_strip<3>, 0, StripGeom<3>::smem);
    if (e == cudaSuccess) e = run(k_sfoc_smooth_strip<5>, 1, StripGeom<5>::smem);
    return e;
}

int smooth_ctas_for(const ImgJob& j, int rows) { return ((j.W + kStW - 1) / kStW) * ((j.H + rows - 1) / rows); }

// Output rows per CTA for one or two images: every CTA streams up to four blocks
// more than it completes, and an SM's time is the blocks of its CTAs (one alone
// runs a block in about half the time of two together): the rows with the
// fewest blocks on the fullest SM.
int strip_rows_for(const ImgJob* j, int n) {
    const long sms = device_sms();
    int H = 0;
    for (int i = 0; i < n; ++i) H = j[i].H > H ? j[i].H : H;
    long best = -1;
    int rows = kStU;
    for (int r = kStU; r < H + kStU; r += kStU) {
        long ctas = 0;
        for (int i = 0; i < n; ++i) ctas += smooth_ctas_for(j[i], r);
        const long cost = (ctas + sms - 1) / sms * (r / kStU + 4);
        if (best < 0 || cost < best) {
            best = cost;
            rows = r;
        }
        if (ctas <= sms) break;  // one CTA per SM already: longer segments only take longer
    }
    return rows;
}

}  // namespace

bool sfoc_batch_supported(const SteerTaps& st, const SmoothTaps& sm) { return steer_is_paper(st) && smooth_is_paper(sm); }

void sfoc_batch_tiles(int H, int W, int* n_steer, int* smooth_ctas) {
    *n_steer = steer_ctas(H, W, steer_rows(H));
    const int rows = strip_rows(H);
    *smooth_ctas = ((W + kStW - 1) / kStW) * ((H + rows - 1) / rows);
}

cudaError_t launch_steer_two(const ImgJob* two, const SteerTaps& st, cudaStream_t s) {
    if (!steer_is_paper(st)) return cudaErrorNotSupported;
    ImgPair p;
    p.j[0] = two[0];
    p.j[1] = two[1];
    const int rows = steer_rows_for(two, 2);
    p.split = steer_ctas(two[0].H, two[0].W, rows);
    k_sfoc_steer_strip<float><<<p.split + steer_ctas(two[1].H, two[1].W, rows), kSrThreads, 0, s>>>(
        p, nullptr, nullptr, 0, st, rows);
    return cudaGetLastError();
}

cudaError_t launch_smooth_two(const ImgJob* two, const SmoothTaps& sm, cudaStream_t s) {
    if (!smooth_is_paper(sm)) return cudaErrorNotSupported;
    ImgPair p;
    p.j[0] = two[0];
    p.j[1] = two[1];
    const int rows = strip_rows_for(two, 2);
    p.split = smooth_ctas_for(two[0], rows);
    return launch_smooth_paper(p, nullptr, nullptr, 0, p.split + smooth_ctas_for(two[1], rows), rows, sm, s);
}

cudaError_t launch_sfoc_batch(const ImgJob* jobs, int n_jobs, const int* steer_begin, int steer_ctas,
                              const int* smooth_begin, int smooth_ctas, const SteerTaps& st, const SmoothTaps& sm,
                              cudaStream_t s) {
    if (n_jobs <= 0) return cudaSuccess;
    if (!sfoc_batch_supported(st, sm)) return cudaErrorNotSupported;
    const ImgPair none = img_none();
    k_sfoc_steer_strip<float><<<steer_ctas, kSrThreads, 0, s>>>(none, jobs, steer_begin, n_jobs, st, 0);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_smooth_paper(none, jobs, smooth_begin, n_jobs, smooth_ctas, 0, sm, s);
}

cudaError_t launch_sfoc_smooth(const float* F, size_t fpitch, int H, int W, const SmoothTaps& tp, Cube& c,
                               cudaStream_t st) {
    dim3 grid((W + kSTW - 1) / kSTW, (H + kSTH - 1) / kSTH);
    cudaError_t e;
    if (smooth_is_paper(tp)) {  // sigma_d 1.0 / 1.5 with rates 1, 2, 3 (Sec. 2.1): one launch per group
        ImgPair pair = img_none();
        ImgJob& one = pair.j[0];
        one.H = H;
        one.W = W;
        one.F = const_cast<float*>(F);
        one.fpitch = fpitch;
        one.c32 = c.f32;
        one.cpitch = c.pitch;
        one.rm = c.rm;
        one.cm = c.cm;
        one.pl = c.pl;
        one.s1 = c.s1;
        one.s2 = c.s2;
        const int rows = strip_rows_for(&one, 1);
        return launch_smooth_paper(pair, nullptr, nullptr, 0, smooth_ctas_for(one, rows), rows, tp, st);
    }
    const int maxhal = tp.halo[0] > tp.halo[1] ? tp.halo[0] : tp.halo[1];
    const int HR = kSTH + 2 * maxhal, FW = smooth_row_stride(maxhal);
    size_t smem = sizeof(float) * ((size_t)HR * FW + (size_t)tp.n_dil * HR * kSTW);
    if (tp.no == 6) {
        e = cudaFuncSetAttribute(k_sfoc_smooth<6>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_sfoc_smooth<6><<<grid, kThreads, smem, st>>>(F, fpitch, fpitch * (size_t)H, H, W, tp, c.f32, c.pitch,
                                                       c.pitch * (size_t)H, c.rm, c.cm, c.pl, c.s1, c.s2);
    } else {
        if (c.rm) return cudaErrorNotSupported;  // bf16 layouts need 12 channels
        e = cudaFuncSetAttribute(k_sfoc_smooth<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_sfoc_smooth<0><<<grid, kThreads, smem, st>>>(F, fpitch, fpitch * (size_t)H, H, W, tp, c.f32, c.pitch,
                                                       c.pitch * (size_t)H, c.rm, c.cm, c.pl, c.s1, c.s2);
    }
    return cudaGetLastError();
}

cudaError_t launch_cube_export(const Cube& c, float* out, cudaStream_t st) {
    const int blocks = 8 * device_sms();
    if (c.dtype == SFOC_DTYPE_BF16)
        k_cube_export_bf16<<<blocks, 256, 0, st>>>(c.rm, c.H, c.W, c.z, out);
    else
        k_cube_export_f32<<<blocks, 256, 0, st>>>(c.f32, c.H, c.W, c.z, c.pitch, out);
    return cudaGetLastError();
}

}  // namespace sfoc

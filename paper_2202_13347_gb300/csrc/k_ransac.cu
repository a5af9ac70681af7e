// Outlier rejection over the control points (Sec. 3.2.3 of arXiv
// 2202.13347): RANSAC with a projective (or affine) model, FP64.
//
//   x' = (h0 x + h1 y + h2) / (h6 x + h7 y + 1),  y' = (h3 x + h4 y + h5) / (h6 x + h7 y + 1)
//   (affine: h6 = h7 = 0).
// Coordinates are normalised first (the valid points' centroid to the
// origin, their mean distance from it to sqrt(2)), every model is solved
// there and mapped back to pixels.  A hypothesis is the exact solution on a
// minimal sample (4 points; affine 3) whose indices the caller supplies (the
// random draws); a singular sample (pivot below 1e-12) scores -1.  The score
// is the number of valid points within `threshold` pixels of the model's
// image; the best score wins, ties to the lower index.  The winner's inliers
// are refitted by least squares (two equations per point, normal equations)
// and recounted, `refits` times.
//
//   k_ransac_frames  one cluster: the two normalising frames (fixed-order sums)
//   k_ransac_solve   8 lanes per hypothesis: the minimal system, a row per lane
//   k_ransac_score   inlier counts of every model: FP32 with an error bound,
//                    FP64 only for points the bound cannot decide
//   k_ransac_final   one cluster: argmax, refits (normal equations reduced in
//                    a fixed order), inlier mask
// FP64 runs at two lanes per clock and SM here (1/64 of FP32), so it sets
// the time of every step that uses it: the steps below either take it off
// the per-(point, hypothesis) path or spread it over more SMs.  1000 points,
// 4096 hypotheses: 556 us before, 115 us now (frames 14, solve 32, score 22, final 45).
#include <cooperative_groups.h>
#include <math.h>

#include <type_traits>

#include "internal.h"

namespace cg = cooperative_groups;

namespace sfoc {

namespace {

constexpr int kRsThreads = 256;
constexpr int kRsCtas = 8;     // CTAs of the cluster of the frame and final kernels (the portable size)
constexpr int kSolveThreads = 32;  // one warp per CTA, so that the warps spread over the SMs
constexpr int kScoreHyps = 16;  // hypotheses per scoring CTA
constexpr int kScorePts = 1024;  // points staged at a time
constexpr int kScoreList = 2048;  // undecided tests listed per CTA and turn (more are decided in place)

struct Frames {
    double s[3];  // source: scale, cx, cy  (p -> s (p - c))
    double d[3];  // destination
    int n_valid;
};

__device__ __forceinline__ bool is_valid(const uint8_t* valid, int i) { return !valid || valid[i] != 0; }

// K sums over the block (fixed order: strided per thread, shuffles, warps in
// order), left in tot[0 .. K-1].  `part`: K doubles per warp.
template <int K>
__device__ void block_sums(double (&v)[K], double* part, double* tot) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    if (l == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) part[w * K + k] = v[k];
    __syncthreads();
    if (threadIdx.x < K) {
        double t = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += part[i * K + threadIdx.x];
        tot[threadIdx.x] = t;
    }
    __syncthreads();
}

// One cluster of kRsCtas CTAs: the two hypot per point are ~50 FP64
// instructions (64 clocks each for a warp), which on a single SM took longer
// than all scoring.  Every CTA takes the means itself; the distances are
// computed in turns of one point per thread of the cluster and added by CTA 0
// in the points' order.
__global__ void __cluster_dims__(kRsCtas, 1, 1) __launch_bounds__(kRsThreads)
    k_ransac_frames(const double* __restrict__ src, const double* __restrict__ dst,
                    const uint8_t* __restrict__ valid, int n, Frames* __restrict__ out) {
    __shared__ double s_part[kRsThreads / 32 * 5], s_tot[5], s_mean[4];
    __shared__ double s_d[2][2][kRsThreads];  // two turns in flight: source and destination distances
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x;
    double a[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int i = tid; i < n; i += kRsThreads)
        if (is_valid(valid, i)) {
            a[0] += 1.0;
            a[1] += src[2 * i];
            a[2] += src[2 * i + 1];
            a[3] += dst[2 * i];
            a[4] += dst[2 * i + 1];
        }
    block_sums(a, s_part, s_tot);
    const double cnt = s_tot[0];
    if (tid < 4) s_mean[tid] = cnt > 0 ? s_tot[1 + tid] / cnt : 0.0;
    __syncthreads();
    const double mx = s_mean[0], my = s_mean[1], nx = s_mean[2], ny = s_mean[3];
    double ds = 0.0, dd = 0.0;
    int turn = 0;
    for (int i0 = 0; i0 < n; i0 += kRsCtas * kRsThreads, turn ^= 1) {
        const int i = i0 + rank * kRsThreads + tid;
        const bool v = i < n && is_valid(valid, i);
        s_d[turn][0][tid] = v ? hypot(src[2 * i] - mx, src[2 * i + 1] - my) : 0.0;
        s_d[turn][1][tid] = v ? hypot(dst[2 * i] - nx, dst[2 * i + 1] - ny) : 0.0;
        // (the next turn's sync orders these reads before this buffer's next use)
        cl.sync();
        if (rank == 0)
            for (int r = 0; r < kRsCtas; ++r) {
                const int j = i0 + r * kRsThreads + tid;
                if (j < n && is_valid(valid, j)) {
                    const double* d = cl.map_shared_rank(&s_d[turn][0][0], r);
                    ds += d[tid];
                    dd += d[kRsThreads + tid];
                }
            }
    }
    cl.sync();  // no CTA leaves while CTA 0 reads its distances
    if (rank != 0) return;
    double d[2] = {ds, dd};
    block_sums(d, s_part, s_tot);
    if (tid < 2) {
        const double mean = cnt > 0 ? s_tot[tid] / cnt : 0.0;
        double* f = tid ? out->d : out->s;
        f[0] = mean > 0.0 ? sqrt(2.0) / mean : 1.0;
        f[1] = s_mean[2 * tid];
        f[2] = s_mean[2 * tid + 1];
    }
    if (tid == 0) out->n_valid = (int)cnt;
}

// the two equations of one correspondence (normalised coordinates)
__device__ __forceinline__ void eq_rows(bool proj, double x, double y, double xp, double yp, double* r1, double* r2) {
    r1[0] = x; r1[1] = y; r1[2] = 1.0; r1[3] = 0.0; r1[4] = 0.0; r1[5] = 0.0;
    r2[0] = 0.0; r2[1] = 0.0; r2[2] = 0.0; r2[3] = x; r2[4] = y; r2[5] = 1.0;
    r1[6] = proj ? -x * xp : 0.0; r1[7] = proj ? -y * xp : 0.0;
    r2[6] = proj ? -x * yp : 0.0; r2[7] = proj ? -y * yp : 0.0;
}

// Gaussian elimination with partial pivoting of one n x n system (n <= 8) by
// a group of 8 lanes: lane r holds row r and right side b, so the divisions
// and updates of a step run side by side (a warp's FP64 instruction takes 64
// clocks whatever its lanes do, and one thread per system needed ~1100 of
// them).  Every lane of the warp calls it; the solution comes back in every
// lane of the group.  False when a pivot falls below 1e-12.
__device__ bool solve_group(double (&A)[8], double b, int n, double (&x)[8]) {
    const unsigned full = 0xffffffffu;
    const int r8 = threadIdx.x & 7;
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        if (c >= n) break;
        int p = c;
        double v = fabs(__shfl_sync(full, A[c], c, 8));
#pragma unroll
        for (int r = c + 1; r < 8; ++r) {
            const double u = fabs(__shfl_sync(full, A[c], r, 8));
            if (r < n && u > v) {
                v = u;
                p = r;
            }
        }
        if (v < 1e-12) ok = false;
        const int from = r8 == c ? p : (r8 == p ? c : r8);
#pragma unroll
        for (int k = c; k < 8; ++k) A[k] = __shfl_sync(full, A[k], from, 8);
        b = __shfl_sync(full, b, from, 8);
        const double f = A[c] / __shfl_sync(full, A[c], c, 8);
        const bool below = r8 > c && r8 < n;
#pragma unroll
        for (int k = c + 1; k < 8; ++k) {
            const double pk = __shfl_sync(full, A[k], c, 8);
            const double up = fma(-f, pk, A[k]);
            A[k] = below && k < n ? up : A[k];
        }
        const double pb = __shfl_sync(full, b, c, 8);
        const double ub = fma(-f, pb, b);
        b = below ? ub : b;
    }
#pragma unroll
    for (int r = 7; r >= 0; --r) {
        x[r] = 0.0;
        if (r >= n) continue;
        double s = b;
#pragma unroll
        for (int k = r + 1; k < 8; ++k)
        {
            const double us = fma(-A[k], x[k], s);
            s = k < n ? us : s;
        }
        x[r] = __shfl_sync(full, s / A[r], r, 8);
    }
    return ok;
}

// Pixel model from the normalised solution (the same in every lane of a group
// of 8): H = Dinv Hn S, scaled to H[8] = 1, with the zeros of Dinv and S left
// out.  *out receives entry (lane mod 8), *last H[8] (1, or NaN where the
// scale is not finite); false when the scale vanishes.
__device__ __forceinline__ bool to_pixels(const double (&h)[8], bool proj, const Frames& F, double* out,
                                          double* last) {
    const double h6 = proj ? h[6] : 0.0, h7 = proj ? h[7] : 0.0;
    const double tx = -F.s[0] * F.s[1], ty = -F.s[0] * F.s[2], di = 1.0 / F.d[0];
    const double M0[3] = {h[0] * F.s[0], h[1] * F.s[0], fma(h[1], ty, h[0] * tx) + h[2]};
    const double M1[3] = {h[3] * F.s[0], h[4] * F.s[0], fma(h[4], ty, h[3] * tx) + h[5]};
    const double M2[3] = {h6 * F.s[0], h7 * F.s[0], fma(h7, ty, h6 * tx) + 1.0};
    const int e = threadIdx.x & 7;
    double mine = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        if (e == j) mine = fma(F.d[1], M2[j], di * M0[j]);
        if (e == 3 + j) mine = fma(F.d[2], M2[j], di * M1[j]);
        if (j < 2 && e == 6 + j) mine = M2[j];
    }
    *out = mine / M2[2];
    *last = isfinite(M2[2]) ? 1.0 : NAN;
    return !(fabs(M2[2]) < 1e-300);
}

__device__ __forceinline__ bool inlier(const double* H, const double* src, const double* dst, int i, double t2) {
    const double x = src[2 * i], y = src[2 * i + 1];
    const double w = H[6] * x + H[7] * y + H[8];
    if (w == 0.0) return false;
    const double ex = (H[0] * x + H[1] * y + H[2]) / w - dst[2 * i];
    const double ey = (H[3] * x + H[4] * y + H[5]) / w - dst[2 * i + 1];
    return ex * ex + ey * ey <= t2;
}

// The minimal systems, a group of 8 lanes per hypothesis (lane r: equation r,
// point r / 2 of the sample).  A singular sample or an index outside [0, n)
// marks its hypothesis with score -1 and a zero model.
__global__ void __launch_bounds__(kSolveThreads)
    k_ransac_solve(const double* __restrict__ src, const double* __restrict__ dst, int n, int proj,
                   const int32_t* __restrict__ samples, int n_hyp, const Frames* __restrict__ frames,
                   int32_t* __restrict__ scores, double* __restrict__ models) {
    const bool pj = proj != 0;
    const int K = pj ? 4 : 3, nu = pj ? 8 : 6;
    const int h = blockIdx.x * (kSolveThreads / 8) + (threadIdx.x >> 3), r8 = threadIdx.x & 7;
    const bool on = h < n_hyp && r8 < nu;
    const Frames F = *frames;
    const int i0 = on ? samples[(size_t)h * K + (r8 >> 1)] : 0;
    const bool in = i0 >= 0 && i0 < n;
    double sx = 0.0, sy = 0.0, dx = 0.0, dy = 0.0;
    if (on && in) {  // an index outside [0, n) voids the hypothesis
        sx = F.s[0] * (src[2 * i0] - F.s[1]);
        sy = F.s[0] * (src[2 * i0 + 1] - F.s[2]);
        dx = F.d[0] * (dst[2 * i0] - F.d[1]);
        dy = F.d[0] * (dst[2 * i0 + 1] - F.d[2]);
    }
    const bool in_range = (__ballot_sync(0xffffffffu, on && !in) >> (threadIdx.x & 24) & 255u) == 0;
    double r1[8], r2[8], A[8], x[8], e, e8;
    eq_rows(pj, sx, sy, dx, dy, r1, r2);
#pragma unroll
    for (int c = 0; c < 8; ++c) A[c] = on ? ((r8 & 1) ? r2[c] : r1[c]) : 0.0;
    bool ok = solve_group(A, (r8 & 1) ? dy : dx, nu, x);
    ok = to_pixels(x, pj, F, &e, &e8) && ok && in_range;
    if (h < n_hyp) {
        models[(size_t)h * 9 + r8] = ok ? e : 0.0;
        if (r8 == 0) {
            models[(size_t)h * 9 + 8] = ok ? e8 : 0.0;
            scores[h] = ok ? 0 : -1;
        }
    }
}

// FP32 decision of the inlier test with an error bound.  A model's FP32 copy
// and the largest |x|, |y|, |x'|, |y'| of the staged points bound the error of
// the mapped position: with u = 2^-24, the numerators and the denominator w
// are within en = 6u (|h0| X + |h1| Y + |h2|) and ew of their exact values,
// so a mapped coordinate is within B = |1/w| (en + m ew) + 8u (m + D) of its
// own (m the larger mapped coordinate, D the largest destination coordinate)
// and the distance to the destination within 2B.  Distances outside the
// threshold -+ 2B are decided; a distance inside, or anything not finite,
// takes the FP64 test, so every decision is the FP64 one.
struct ModelF {
    float h[9];
    float en, ew;
};
struct PointF {
    float x, y, dx, dy;
};
constexpr float kU6 = 6.f * 5.9604645e-8f, kU8 = 8.f * 5.9604645e-8f;

__device__ __forceinline__ ModelF model_f(const double* H, float X, float Y) {
    ModelF m;
#pragma unroll
    for (int r = 0; r < 9; ++r) m.h[r] = (float)H[r];
    m.en = kU6 * 1.01f * fmaxf(fabsf(m.h[0]) * X + fabsf(m.h[1]) * Y + fabsf(m.h[2]),
                               fabsf(m.h[3]) * X + fabsf(m.h[4]) * Y + fabsf(m.h[5]));
    m.ew = kU6 * 1.01f * (fabsf(m.h[6]) * X + fabsf(m.h[7]) * Y + fabsf(m.h[8]));
    return m;
}

// 1: inlier, 0: not, -1: undecided.  T: the threshold (at most kMaxFastT).
constexpr float kMaxFastT = 1e6f;
__device__ __forceinline__ int inlier_f(const ModelF& m, const PointF& p, float D, float T) {
    const float w = fmaf(m.h[6], p.x, fmaf(m.h[7], p.y, m.h[8]));
    const float r = 1.f / w;
    const float px = fmaf(m.h[0], p.x, fmaf(m.h[1], p.y, m.h[2])) * r;
    const float py = fmaf(m.h[3], p.x, fmaf(m.h[4], p.y, m.h[5])) * r;
    const float ex = px - p.dx, ey = py - p.dy;
    const float d2 = fmaf(ex, ex, ey * ey);
    const float mm = fmaxf(fabsf(px), fabsf(py));
    // the error of w may not reach a tenth of it, so that 1/w is good to first order
    const float B2 = 2.4f * fmaf(fabsf(r), fmaf(mm, m.ew, m.en), kU8 * (mm + D));
    const float hi = T + B2, lo = T - B2;
    if (!(m.ew < 0.1f * fabsf(w))) return -1;
    if (d2 * 0.999999f > hi * hi) return 0;
    if (lo > 0.f && d2 * 1.000001f < lo * lo) return 1;
    return -1;
}

// Inlier counts: one warp per two of the CTA's kScoreHyps models, the points
// staged as FP32 once per CTA.  4096 hypotheses over 1000 points are 4.1M
// tests of ~45 FP32 instructions; with FP64 (two divisions a test) they took
// most of the call.  The undecided tests (within ~0.01 px of the threshold)
// are listed and taken together: one undecided lane would hold its warp for a
// whole FP64 test (~3000 clocks).
__global__ void __launch_bounds__(kRsThreads)
    k_ransac_score(const double* __restrict__ src, const double* __restrict__ dst, const uint8_t* __restrict__ valid,
                   int n, int n_hyp, double t2, float T, int32_t* __restrict__ scores,
                   const double* __restrict__ models) {
    constexpr int kWarps = kRsThreads / 32, kPer = kScoreHyps / kWarps;
    __shared__ float4 s_p[kScorePts];  // x, y, x', y'; x' = +inf: not valid (decided as an outlier)
    __shared__ float s_mx[kWarps][3];
    __shared__ unsigned s_undec[kScoreList];  // undecided tests: model * kScorePts + point
    __shared__ int s_nu, s_extra[kScoreHyps];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < kScoreHyps) s_extra[threadIdx.x] = 0;
    int cnt[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) cnt[q] = 0;
    for (int i0 = 0; i0 < n; i0 += kScorePts) {
        const int np = min(kScorePts, n - i0);
        float X = 0.f, Y = 0.f, D = 0.f;
        __syncthreads();  // the previous points are done with
        if (threadIdx.x == 0) s_nu = 0;
        for (int i = threadIdx.x; i < np; i += kRsThreads) {
            const bool v = is_valid(valid, i0 + i);
            const double* a = src + 2 * (size_t)(i0 + i);
            const double* b = dst + 2 * (size_t)(i0 + i);
            const float4 p = v ? make_float4((float)a[0], (float)a[1], (float)b[0], (float)b[1])
                               : make_float4(0.f, 0.f, INFINITY, 0.f);
            s_p[i] = p;
            if (v) {
                X = fmaxf(X, fabsf(p.x));
                Y = fmaxf(Y, fabsf(p.y));
                D = fmaxf(D, fmaxf(fabsf(p.z), fabsf(p.w)));
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            X = fmaxf(X, __shfl_xor_sync(0xffffffffu, X, o));
            Y = fmaxf(Y, __shfl_xor_sync(0xffffffffu, Y, o));
            D = fmaxf(D, __shfl_xor_sync(0xffffffffu, D, o));
        }
        if (lane == 0) {
            s_mx[w][0] = X;
            s_mx[w][1] = Y;
            s_mx[w][2] = D;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kWarps; ++q) {
            X = fmaxf(X, s_mx[q][0]);
            Y = fmaxf(Y, s_mx[q][1]);
            D = fmaxf(D, s_mx[q][2]);
        }
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int h = blockIdx.x * kScoreHyps + w * kPer + q;
            if (h >= n_hyp || scores[h] < 0) continue;
            const double* Hg = models + (size_t)h * 9;
            const ModelF m = model_f(Hg, X, Y);
            // four points at a time, so that their divisions overlap
            for (int i4 = lane; i4 < np; i4 += 4 * 32) {
                int in[4];
                bool und = false;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = i4 + 32 * u;
                    const float4 p = s_p[i < np ? i : 0];
                    in[u] = i < np ? inlier_f(m, PointF{p.x, p.y, p.z, p.w}, D, T) : 0;
                    und = und || in[u] < 0;
                    cnt[q] += max(in[u], 0);
                }
                if (!und) continue;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (in[u] >= 0) continue;
                    const int i = i4 + 32 * u, at = atomicAdd(&s_nu, 1);
                    if (at < kScoreList) s_undec[at] = (unsigned)((w * kPer + q) * kScorePts + i);
                    else cnt[q] += is_valid(valid, i0 + i) && inlier(Hg, src, dst, i0 + i, t2) ? 1 : 0;
                }
            }
        }
        __syncthreads();
        const int nu = min(s_nu, kScoreList);
        for (int u = threadIdx.x; u < nu; u += kRsThreads) {
            const int q = (int)(s_undec[u] / kScorePts), i = i0 + (int)(s_undec[u] % kScorePts);
            if (is_valid(valid, i) && inlier(models + (size_t)(blockIdx.x * kScoreHyps + q) * 9, src, dst, i, t2))
                atomicAdd(&s_extra[q], 1);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int h = blockIdx.x * kScoreHyps + w * kPer + q;
        int c = cnt[q];
        for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
        if (lane == 0 && h < n_hyp && scores[h] >= 0) scores[h] = c + s_extra[w * kPer + q];
    }
}

constexpr int kNE = 44;  // unique entries of the 8 x 8 normal matrix (36) and the right side (8)

// One cluster of kRsCtas CTAs, the points strided over them: a single SM's
// FP64 unit held the recounts and the normal equations for longer than the
// scoring of every hypothesis takes.  Each thread's 44 sums go through shared
// memory (a shuffle tree would run its FP64 adds with idle lanes), then over
// the CTAs in order; warp 0 of every CTA solves the same system.
struct FinalSmem {
    double e[kNE][kRsThreads + 1];
    double tot[kNE];
};

__global__ void __cluster_dims__(kRsCtas, 1, 1) __launch_bounds__(kRsThreads)
    k_ransac_final(const double* __restrict__ src, const double* __restrict__ dst, const uint8_t* __restrict__ valid,
                   int n, int proj, int n_hyp, double t2, int refits, const Frames* __restrict__ frames,
                   const int32_t* __restrict__ scores, const double* __restrict__ models, double* __restrict__ H_out,
                   uint8_t* __restrict__ mask, int32_t* __restrict__ info) {
    extern __shared__ __align__(16) char fin_sm[];
    FinalSmem& S = *reinterpret_cast<FinalSmem*>(fin_sm);
    __shared__ int s_best, s_score[kRsThreads / 32], s_idx[kRsThreads / 32];
    __shared__ double sH[9];
    __shared__ int s_cnt[kRsThreads / 32];
    __shared__ int s_total;  // this CTA's inlier count (read by the others)
    __shared__ int s_ok;
    cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int first = (int)cl.block_rank() * kRsThreads + tid, step = kRsCtas * kRsThreads;
    const bool pj = proj != 0;
    const int k = pj ? 4 : 3, nu = pj ? 8 : 6;
    // argmax: highest score, then lowest index (every CTA over all of them)
    auto take = [](int s, int i, int& bs, int& bi) {
        if (i >= 0 && (bi < 0 || s > bs || (s == bs && i < bi))) {
            bs = s;
            bi = i;
        }
    };
    int bs = -2, bi = -1;
    for (int h = tid; h < n_hyp; h += kRsThreads) take(scores[h], h, bs, bi);
    for (int o = 16; o > 0; o >>= 1) {
        const int os = __shfl_down_sync(0xffffffffu, bs, o), oi = __shfl_down_sync(0xffffffffu, bi, o);
        take(os, oi, bs, bi);
    }
    if (lane == 0) {
        s_score[w] = bs;
        s_idx[w] = bi;
    }
    __syncthreads();
    if (tid == 0) {
        for (int t = 1; t < kRsThreads / 32; ++t) take(s_score[t], s_idx[t], bs, bi);
        s_best = bi >= 0 && bs >= 0 ? bi : -1;  // every hypothesis singular: no winner
        for (int q = 0; q < 9; ++q) sH[q] = s_best >= 0 ? models[(size_t)s_best * 9 + q] : ((q % 4 == 0) ? 1.0 : 0.0);
    }
    __syncthreads();
    const int best = s_best;
    auto recount = [&]() -> int {
        double H[9];
        for (int q = 0; q < 9; ++q) H[q] = sH[q];
        int c = 0;
        for (int i = first; i < n; i += step) {
            const bool in = best >= 0 && is_valid(valid, i) && inlier(H, src, dst, i, t2);
            mask[i] = in ? 1 : 0;
            c += in ? 1 : 0;
        }
        for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
        if (lane == 0) s_cnt[w] = c;
        __syncthreads();
        if (tid == 0) {
            int t = 0;
            for (int q = 0; q < kRsThreads / 32; ++q) t += s_cnt[q];
            s_total = t;
        }
        cl.sync();
        int t = 0;
        for (unsigned r = 0; r < cl.num_blocks(); ++r) t += *cl.map_shared_rank(&s_total, r);
        cl.sync();  // read by every CTA before the next count (or a CTA leaves)
        return t;
    };
    int cnt = recount();
    const Frames F = *frames;
    const int rows = n - (int)cl.block_rank() * kRsThreads;  // threads of this CTA with a point
    const int act = rows < 0 ? 0 : (rows < kRsThreads ? rows : kRsThreads);
    for (int it = 0; it < refits && best >= 0 && cnt >= k; ++it) {
        // normal equations over this thread's inliers (the mask it wrote itself)
        double e[kNE];
#pragma unroll
        for (int q = 0; q < kNE; ++q) e[q] = 0.0;
        for (int i = first; i < n; i += step) {
            if (!mask[i]) continue;
            double r1[8], r2[8];
            const double sx = F.s[0] * (src[2 * i] - F.s[1]), sy = F.s[0] * (src[2 * i + 1] - F.s[2]);
            const double dx = F.d[0] * (dst[2 * i] - F.d[1]), dy = F.d[0] * (dst[2 * i + 1] - F.d[2]);
            eq_rows(pj, sx, sy, dx, dy, r1, r2);
            int q = 0;
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int c = a; c < 8; ++c) {
                    // the zero entries of the two rows add nothing (columns 0-2 of
                    // the second, 3-5 of the first)
                    if (c < 3) e[q] += r1[a] * r1[c];
                    else if (a < 3 && c < 6) e[q] += 0.0;
                    else if (a < 3) e[q] += r1[a] * r1[c];
                    else if (a < 6) e[q] += r2[a] * r2[c];
                    else e[q] += r1[a] * r1[c] + r2[a] * r2[c];
                    ++q;
                }
#pragma unroll
            for (int a = 0; a < 8; ++a) e[q++] += a < 3 ? r1[a] * dx : (a < 6 ? r2[a] * dy : r1[a] * dx + r2[a] * dy);
        }
#pragma unroll
        for (int q = 0; q < kNE; ++q) S.e[q][tid] = e[q];
        __syncthreads();
        {
            // four threads per entry, a quarter of the rows each, then in order
            const int q = tid >> 2, part = tid & 3;
            double v = 0.0;
            if (q < kNE)
                for (int r = part * (kRsThreads / 4); r < min((part + 1) * (kRsThreads / 4), act); ++r) v += S.e[q][r];
            const double v1 = __shfl_down_sync(0xffffffffu, v, 1), v2 = __shfl_down_sync(0xffffffffu, v, 2),
                         v3 = __shfl_down_sync(0xffffffffu, v, 3);
            if (q < kNE && part == 0) S.tot[q] = ((v + v1) + v2) + v3;
        }
        cl.sync();
        if (w == 0) {
            double tot[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int q = lane + 32 * u;
                tot[u] = 0.0;
                if (q < kNE)
                    for (unsigned r = 0; r < cl.num_blocks(); ++r) tot[u] += cl.map_shared_rank(&S, r)->tot[q];
            }
            // lane r takes row r of the symmetric matrix (entry (a, c >= a) at a (17 - a) / 2 + c - a)
            auto entry = [&](int q) {
                const double lo = __shfl_sync(0xffffffffu, tot[0], q & 31), hi = __shfl_sync(0xffffffffu, tot[1], q & 31);
                return q < 32 ? lo : hi;
            };
            const int r = lane & 7;
            double M[8], x[8], mine, last;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int a = min(r, c), b = max(r, c);
                M[c] = entry(a * (17 - a) / 2 + b - a);
            }
            const double rhs = entry(36 + r);
            bool ok = solve_group(M, rhs, nu, x);
            ok = to_pixels(x, pj, F, &mine, &last) && ok;
            if (lane == 0) s_ok = ok;
            if (ok && lane < 8) sH[lane] = mine;
            if (ok && lane == 8) sH[8] = last;
        }
        cl.sync();  // S.tot read by every CTA; sH written
        if (!s_ok) break;  // the same in every CTA
        cnt = recount();
    }
    if (first == 0) {
        for (int q = 0; q < 9; ++q) H_out[q] = sH[q];
        info[0] = best;
        info[1] = best >= 0 ? cnt : 0;
    }
}

// Rectification (Sec. 3.2.3): out(x, y) = bilinear sample of the sensed
// image at H^-1 (x, y); outside [0, W-1] x [0, H-1] the fill value.  Each CTA
// inverts H (the adjugate scaled by its last entry); a singular model gives
// an all-fill image.  The mapping is as good as FP64 (coordinates of 10^4 px
// keep their sub-pixel part), the blend FP32.
//
// FP64 runs at two lanes per clock and SM, so the mapping of every pixel in
// FP64 (~50 instructions) set the time: 2048 x 2048 took 349 us against 5 us
// of HBM time.  Here a warp maps one pixel of its kRectW x kRectH tile in
// FP64, (u0, t0) at (x0, y0), and steps from it exactly:
//   u(x0 + i, y0 + k) = u0 + d / (1 + e),  d = i sx + k sy,  e = i qx + k qy,
//   sx = (a - g u0) / w0, sy = (b - h u0) / w0, qx = g / w0, qy = h / w0
// (a, b, g, h the model's x row and its last row).  Positions and steps are
// 64-bit integers in 2^-32 px, so that u0 + d is exact but for the steps'
// roundings (at most 40 x 2^-33 px); the rest, -d e / (1 + e), is below 1/16 px
// on the tiles that take this route and comes from FP32 with at most
// 9 x 2^-24 of its size in error.  A position is thus within 2^-24 px of the FP64
// one wherever it lies (2^-27 without perspective), and its fraction is rounded
// to FP32 once, as after the FP64 mapping: the values of a noise image are
// 1.94e-8 rms from float64 either way.  (With FP32 fractions added up they were
// 3.4e-8, positions up to 2^-22 px off, and the call no faster: 2048 x 2048 25.4
// us, with this 25.1.)
// Tiles with a strong perspective or scale, and pixels mapped within 2^-10 px of
// the image's border lines (where a rounding could decide inside or outside),
// take the FP64 mapping itself.  Tiles well inside the image (most) skip the
// border tests.
// The CTA's first warp prepares up to 32 tiles, one per lane (inverse, tile
// maps: a chain of ~1500 clocks whose length does not depend on their
// number), so large images give a warp four tiles (kRectTiles) and small ones
// one, which keeps more CTAs.
constexpr int kRectW = 32, kRectH = 8, kRectTiles = 4, kRectB = 4;
typedef unsigned long long u64;
struct RectTile {
    u64 p[2], sx[2], sy[2];     // per axis (u, t): position of the tile's first pixel and steps, 2^-32 px
    float fsx[2], fsy[2];       // the steps
    float qx, qy;
    int ok;                     // the steps serve the whole tile: 2 if all of it maps at least a pixel inside
                                // the image's border lines, else 1
};

// one pixel by the FP64 mapping
__device__ __noinline__ float rect_fp64(const float* __restrict__ img, int H, int W, size_t pitch, const double* inv,
                                        int ok, int x, int y, float fill) {
    const double w = inv[6] * x + inv[7] * y + inv[8];
    if (!ok || w == 0.0) return fill;
    const double rw = 1.0 / w;
    const double u = (inv[0] * x + inv[1] * y + inv[2]) * rw;
    const double t = (inv[3] * x + inv[4] * y + inv[5]) * rw;
    if (!(u >= 0.0 && t >= 0.0 && u <= W - 1 && t <= H - 1)) return fill;
    const int u0 = min((int)floor(u), max(W - 2, 0)), t0 = min((int)floor(t), max(H - 2, 0));
    const int u1 = min(u0 + 1, W - 1), t1 = min(t0 + 1, H - 1);
    const float fu = (float)(u - u0), ft = (float)(t - t0);
    const float p00 = img[(size_t)t0 * pitch + u0], p01 = img[(size_t)t0 * pitch + u1];
    const float p10 = img[(size_t)t1 * pitch + u0], p11 = img[(size_t)t1 * pitch + u1];
    const float r0 = fmaf(fu, p01 - p00, p00), r1 = fmaf(fu, p11 - p10, p10);
    return fmaf(ft, r1 - r0, r0);
}

// One column of a tile.  INSIDE: every pixel samples inside the image.
template <bool INSIDE>
__device__ __forceinline__ void rect_tile(const float* __restrict__ img, int H, int W, size_t pitch, const RectTile& T,
                                          const double* s_inv, int s_ok, float fill, int x, int y0, int lane, int out_h,
                                          int out_w, float* __restrict__ out) {
    constexpr int kB = INSIDE ? kRectB : 2;  // (the general form holds twice as much per row)
    const float fi = (float)lane;
    // inside, samples are addressed by 32-bit offsets from the tile's first one
    const float* const base = INSIDE ? img + (size_t)(T.p[1] >> 32) * pitch + (size_t)(T.p[0] >> 32) : img;
    u64 pos[2];   // this column at the current row
    float dx[2];  // its steps from the tile's first pixel
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        pos[q] = (INSIDE ? T.p[q] & 0xffffffffull : T.p[q]) + (u64)lane * T.sx[q];
        dx[q] = fi * T.fsx[q];
    }
    // kB rows at a time: their positions, then all their samples in flight,
    // then the blends (with one row after the other the kernel waited for every
    // row's samples: 60 us)
#pragma unroll 1
    for (int kb = 0; kb < kRectH; kb += kB) {
        if (y0 + kb >= out_h) break;
        typename std::conditional<INSIDE, int, size_t>::type at[kB];
        float fu[kB], ft[kB];
        bool ld[kB], fp64[kB];
        bool any64 = false;
#pragma unroll
        for (int b = 0; b < kB; ++b) {
            const float fk = (float)(kb + b);
            const float e0 = fmaf(fi, T.qx, fk * T.qy);
            const float e = e0 * (1.f - e0 * (1.f - e0));  // e0 / (1 + e0), e0 < 2^-10
            int ci[2];
            float fr[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float c = -e * fmaf(fk, T.fsy[q], dx[q]);  // the perspective term
                const u64 at64 = pos[q] + (u64)(long long)__float2int_rn(c * 4294967296.f);
                pos[q] += T.sy[q];
                ci[q] = (int)(at64 >> 32);
                fr[q] = __uint2float_rn((unsigned)at64) * (1.f / 4294967296.f);
            }
            ld[b] = true;
            if (!INSIDE) {
                // inside, outside, or within 2^-10 px of the image's border lines, where
                // the FP64 mapping decides
                ld[b] = T.ok != 0;
                fp64[b] = T.ok == 0;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int last = (q ? H : W) - 1;
                    constexpr float eps = 1.f / 1024;
                    fp64[b] = fp64[b] || (fr[q] < eps && (ci[q] == 0 || ci[q] == last)) ||
                              (fr[q] > 1.f - eps && (ci[q] == -1 || ci[q] == last - 1));
                    ld[b] = ld[b] && ci[q] >= 0 && ci[q] < last;
                }
                any64 = any64 || fp64[b];
            }
            if (INSIDE) at[b] = ci[1] * (int)pitch + ci[0];
            else at[b] = ld[b] ? (size_t)ci[1] * pitch + ci[0] : 0;
            fu[b] = fr[0];
            ft[b] = fr[1];
        }
        float p00[kB], p01[kB], p10[kB], p11[kB];
#pragma unroll
        for (int b = 0; b < kB; ++b) {
            const float *r0 = base + at[b], *r1 = r0 + pitch;
            p00[b] = ld[b] ? r0[0] : 0.f;
            p01[b] = ld[b] ? r0[1] : 0.f;
            p10[b] = ld[b] ? r1[0] : 0.f;
            p11[b] = ld[b] ? r1[1] : 0.f;
        }
        float* const o = out + (size_t)(y0 + kb) * out_w + x;
#pragma unroll
        for (int b = 0; b < kB; ++b) {
            const float r0 = fmaf(fu[b], p01[b] - p00[b], p00[b]), r1 = fmaf(fu[b], p11[b] - p10[b], p10[b]);
            if (y0 + kb + b < out_h) o[(size_t)b * out_w] = ld[b] ? fmaf(ft[b], r1 - r0, r0) : fill;
        }
        if (!INSIDE && any64) {
            for (int b = 0; b < kB; ++b) {
                const int y = y0 + kb + b;
                bool mine = false;
#pragma unroll
                for (int u = 0; u < kB; ++u) mine = mine || (u == b && fp64[u]);
                if (mine && y < out_h) out[(size_t)y * out_w + x] = rect_fp64(img, H, W, pitch, s_inv, s_ok, x, y, fill);
            }
        }
    }
}

__global__ void __launch_bounds__(kRsThreads, 4)
    k_rectify(const float* __restrict__ img, int H, int W, size_t pitch, const double* __restrict__ Hm, float fill,
              int out_h, int out_w, float* __restrict__ out, int per_warp) {
    constexpr int kWarps = kRsThreads / 32;
    __shared__ double s_inv[9];
    __shared__ int s_ok;
    __shared__ RectTile s_tile[kWarps * kRectTiles];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // tile t of the CTA (t < kWarps * per_warp): column block t / kWarps, row block t % kWarps
    const int xb = blockIdx.x * kRectW * per_warp, yb = blockIdx.y * (kRectH * kWarps);
    // a warp's FP64 instruction holds its sub-partition's FP64 unit for 64
    // clocks: neighbouring CTAs use different warps for this
    if (warp == (int)((blockIdx.x + blockIdx.y) & (kWarps - 1))) {
        {
            const double a = Hm[0], b = Hm[1], c = Hm[2], d = Hm[3], e = Hm[4], f = Hm[5], g = Hm[6], h = Hm[7],
                         i = Hm[8];
            const double inv[9] = {e * i - f * h, c * h - b * i, b * f - c * e, f * g - d * i, a * i - c * g,
                                   c * d - a * f, d * h - e * g, b * g - a * h, a * e - b * d};
            const double det = a * inv[0] + b * inv[3] + c * inv[6];
            const bool ok = det != 0.0 && inv[8] != 0.0;
            double mine = inv[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (lane == k) mine = inv[k];
            if (lane < 9) s_inv[lane] = ok ? mine / inv[8] : 0.0;
            if (lane == 0) s_ok = ok;
        }
        __syncwarp();
        if (lane < kWarps * per_warp) {  // lane t: tile t
            RectTile T;
            const double x = xb + (lane / kWarps) * kRectW, y = yb + (lane % kWarps) * kRectH;
            const double w = s_inv[6] * x + s_inv[7] * y + s_inv[8];
            const double rw = 1.0 / w;
            const double p[2] = {(s_inv[0] * x + s_inv[1] * y + s_inv[2]) * rw,
                                 (s_inv[3] * x + s_inv[4] * y + s_inv[5]) * rw};
            const double qx = s_inv[6] * rw, qy = s_inv[7] * rw;
            bool ok = s_ok && fabs(p[0]) < 1e8 && fabs(p[1]) < 1e8 &&
                      fabs(qx) * kRectW + fabs(qy) * kRectH < 1.0 / 1024;
            T.qx = (float)qx;
            T.qy = (float)qy;
            const float reach = fabsf(T.qx) * (kRectW - 1) + fabsf(T.qy) * (kRectH - 1);  // the largest |e|
            constexpr double k32 = 4294967296.0;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const double sx = (s_inv[3 * q] - s_inv[6] * p[q]) * rw, sy = (s_inv[3 * q + 1] - s_inv[7] * p[q]) * rw;
                T.fsx[q] = (float)sx;
                T.fsy[q] = (float)sy;
                ok = ok && fabs(sx) < 4.0 && fabs(sy) < 4.0 &&
                     (fabsf(T.fsx[q]) * (kRectW - 1) + fabsf(T.fsy[q]) * (kRectH - 1)) * reach < 1.f / 16;
                T.p[q] = (u64)__double2ll_rn(p[q] * k32);
                T.sx[q] = (u64)__double2ll_rn(sx * k32);
                T.sy[q] = (u64)__double2ll_rn(sy * k32);
            }
            // how far the tile reaches to either side, with 1 % for the perspective
            bool in = ok && pitch < ((size_t)1 << 23);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float c = (float)p[q], last = (float)((q ? H : W) - 1);
                const float ex = (kRectW - 1) * T.fsx[q], ey = (kRectH - 1) * T.fsy[q];
                in = in && c + 1.01f * (fminf(ex, 0.f) + fminf(ey, 0.f)) > 2.f &&
                     c + 1.01f * (fmaxf(ex, 0.f) + fmaxf(ey, 0.f)) < last - 2.f && last < 4194304.f;
            }
            T.ok = in ? 2 : ok ? 1 : 0;
            s_tile[lane] = T;
        }
    }
    __syncthreads();
    for (int xt = 0; xt < per_warp; ++xt) {
        const int x = xb + xt * kRectW + lane, y0 = yb + warp * kRectH;
        if (x >= out_w) break;
        const RectTile& T = s_tile[xt * kWarps + warp];
        if (T.ok == 2) rect_tile<true>(img, H, W, pitch, T, s_inv, s_ok, fill, x, y0, lane, out_h, out_w, out);
        else rect_tile<false>(img, H, W, pitch, T, s_inv, s_ok, fill, x, y0, lane, out_h, out_w, out);
    }
}

__global__ void k_results_to_points(const int32_t* __restrict__ pts, const fastncc_result* __restrict__ res, int n,
                                    double* __restrict__ src, double* __restrict__ dst, uint8_t* __restrict__ valid) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const fastncc_result r = res[i];
    const double x = pts[2 * i], y = pts[2 * i + 1];
    src[2 * i] = x;
    src[2 * i + 1] = y;
    dst[2 * i] = x + (double)r.sub_dx;  // the refined offset (dx plus its parabola correction)
    dst[2 * i + 1] = y + (double)r.sub_dy;
    valid[i] = r.status == SFOC_PT_OK ? 1 : 0;
}

}  // namespace

size_t ransac_workspace_bytes(int n_hyp) {
    return (sizeof(Frames) + 255) / 256 * 256 + (sizeof(int32_t) * (size_t)n_hyp + 255) / 256 * 256 +
           sizeof(double) * 9 * (size_t)n_hyp;
}

cudaError_t launch_ransac(const double* src, const double* dst, const uint8_t* valid, int n, int proj,
                          const int32_t* samples, int n_hyp, double threshold, int refits, double* H_out,
                          uint8_t* mask, int32_t* info, int32_t* scores_out, void* ws, cudaStream_t st, int* launches) {
    char* p = static_cast<char*>(ws);
    Frames* frames = reinterpret_cast<Frames*>(p);
    p += (sizeof(Frames) + 255) / 256 * 256;
    int32_t* scores = scores_out ? scores_out : reinterpret_cast<int32_t*>(p);
    p += (sizeof(int32_t) * (size_t)n_hyp + 255) / 256 * 256;
    double* models = reinterpret_cast<double*>(p);
    const double t2 = threshold * threshold;
    // the FP32 decision serves thresholds well inside its range; beyond, T = NaN
    // leaves every point undecided and the FP64 test decides
    const float T = threshold <= (double)kMaxFastT ? (float)threshold : NAN;
    k_ransac_frames<<<kRsCtas, kRsThreads, 0, st>>>(src, dst, valid, n, frames);
    int nl = 1;
    if (n_hyp > 0) {
        const int sb = (n_hyp + kSolveThreads / 8 - 1) / (kSolveThreads / 8);
        k_ransac_solve<<<sb, kSolveThreads, 0, st>>>(src, dst, n, proj, samples, n_hyp, frames, scores, models);
        k_ransac_score<<<(n_hyp + kScoreHyps - 1) / kScoreHyps, kRsThreads, 0, st>>>(src, dst, valid, n, n_hyp, t2, T,
                                                                                     scores, models);
        nl += 2;
    }
    const int smem = (int)sizeof(FinalSmem);
    cudaError_t e = cudaFuncSetAttribute(k_ransac_final, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_ransac_final<<<kRsCtas, kRsThreads, smem, st>>>(src, dst, valid, n, proj, n_hyp, t2, refits, frames, scores,
                                                      models, H_out, mask, info);
    ++nl;
    if (launches) *launches = nl;
    return cudaGetLastError();
}

cudaError_t launch_rectify(const float* img, int H, int W, size_t pitch, const double* Hm, float fill, int out_h,
                           int out_w, float* out, cudaStream_t st) {
    constexpr int rows = kRectH * (kRsThreads / 32);
    const unsigned gy = (unsigned)((out_h + rows - 1) / rows);
    // four tiles a warp once that still leaves two CTAs per SM
    const int per = (size_t)gy * ((out_w + kRectTiles * kRectW - 1) / (kRectTiles * kRectW)) >= 2 * (size_t)device_sms()
                        ? kRectTiles
                        : 1;
    dim3 grid((unsigned)((out_w + per * kRectW - 1) / (per * kRectW)), gy);
    k_rectify<<<grid, kRsThreads, 0, st>>>(img, H, W, pitch, Hm, fill, out_h, out_w, out, per);
    return cudaGetLastError();
}

cudaError_t launch_results_to_points(const int32_t* pts, const fastncc_result* res, int n, double* src, double* dst,
                                     uint8_t* valid, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_results_to_points<<<(n + 255) / 256, 256, 0, st>>>(pts, res, n, src, dst, valid);
    return cudaGetLastError();
}

}  // namespace sfoc

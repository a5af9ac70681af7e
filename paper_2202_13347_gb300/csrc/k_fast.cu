// Block-based FAST interest points (Sec. 3.1.1 of arXiv 2202.13347): the
// FAST operator per block of a partition of the image, so that the points
// spread evenly.
//
// Segment test FAST-9 on the 16 pixels of the radius-3 circle; the score of
// a pixel is the largest threshold for which it is still a corner (the
// largest over the 16 arcs of 9 contiguous circle pixels of the arc's
// smallest difference to the centre, brighter or darker), taken in FP32 as
// the image is stored; it is a corner when the score exceeds t.  Pixels
// closer than 3 to the border score 0.  A corner survives 3 x 3
// non-maximum suppression when its score is at least every neighbour's and
// above those before it in raster order.  Each block (grid_y x grid_x
// partition, rows [by H / grid_y, (by + 1) H / grid_y), columns likewise)
// keeps its strongest surviving corner at least `margin` from the border,
// ties to the smaller y, then x.
//
// One CTA per block, walking the block in sub-tiles of up to 64 x 64
// outputs: the image with a 4-pixel halo is staged in shared memory; every
// pixel of the sub-tile and a 1-pixel ring (for the suppression) takes a
// quick test, the pixels that pass it are listed and scored, and the listed
// pixels inside the sub-tile take the suppression; then each thread keeps
// its best candidate and the CTA reduces.
// Quick test: an arc of 9 of the 16 circle pixels holds one pixel of every
// opposite pair (k, k + 8), so a pixel is no corner when both pixels of some
// pair are at most t brighter and both of some pair at most t darker.  Four
// pairs (8 of the 16 differences) turn away most pixels, whose score is 0
// either way, and the list keeps the full score's warps dense: the score is
// ~180 FP32 operations a pixel and set the time of the kernel (2048 x 2048,
// 32 x 32 blocks: 59 us before, 25 us with the quick test).
#include "internal.h"

namespace sfoc {

namespace {

constexpr int kFastThreads = 256;
constexpr int kSub = 64;             // outputs per sub-tile side
constexpr int kIn = kSub + 8;        // staged image side (4-pixel halo)
constexpr int kSc = kSub + 2;        // scores side (1-pixel ring)

// circle pixel k, clockwise from the top (k is a constant wherever these are unrolled)
__device__ __forceinline__ constexpr int cdx(int k) {
    constexpr int v[16] = {0, 1, 2, 3, 3, 3, 2, 1, 0, -1, -2, -3, -3, -3, -2, -1};
    return v[k];
}
__device__ __forceinline__ constexpr int cdy(int k) { return -cdx((k + 4) & 15); }

// candidate order: higher score, then smaller y, then smaller x
__device__ __forceinline__ bool better(float s, int y, int x, float bs, int by, int bx) {
    if (bx < 0) return x >= 0;
    if (x < 0) return false;
    if (s != bs) return s > bs;
    return y < by || (y == by && x < bx);
}

// the score of the pixel at staged position (iy, ix), 0 where it is no corner
__device__ __forceinline__ float fast_score(const float (*s_img)[kIn + 1], int iy, int ix, float t) {
    const float c = s_img[iy][ix];
    float d[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) d[k] = s_img[iy + cdy(k)][ix + cdx(k)] - c;
    // smallest and largest difference over every arc of 9 (cyclic),
    // by doubling: windows of 2, 4, 8, then one more pixel
    float lo[16], hi[16], l2[16], h2[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        lo[k] = fminf(d[k], d[(k + 1) & 15]);
        hi[k] = fmaxf(d[k], d[(k + 1) & 15]);
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        l2[k] = fminf(lo[k], lo[(k + 2) & 15]);
        h2[k] = fmaxf(hi[k], hi[(k + 2) & 15]);
    }
    float bright = -INFINITY, dark = INFINITY;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float mn = fminf(fminf(l2[k], l2[(k + 4) & 15]), d[(k + 8) & 15]);
        const float mx = fmaxf(fmaxf(h2[k], h2[(k + 4) & 15]), d[(k + 8) & 15]);
        bright = fmaxf(bright, mn);   // brighter arc: its smallest rise
        dark = fminf(dark, mx);       // darker arc: minus its smallest drop
    }
    const float best = fmaxf(bright, -dark);
    return best > t ? best : 0.f;
}

// QUICK: the quick test first.  Without it (a threshold of 0, which turns away
// nothing but flat pixels) every pixel is scored and the corners are listed: 2048 x
// 2048 texture, threshold 0, blocks of 512 x 512 1163 us with the test, 1010 without,
// of 64 x 64 77 and 67.  (Scoring at once the pixels of a warp that passes mostly,
// or a sub-tile after one that did, made the usual thresholds 3 to 15 % slower.)
template <bool QUICK>
__global__ void __launch_bounds__(kFastThreads)
    k_fast_blocks(const float* __restrict__ img, int H, int W, size_t pitch, float t, int grid_y, int grid_x,
                  int margin, int32_t* __restrict__ points, float* __restrict__ scores) {
    __shared__ float s_img[kIn][kIn + 1];
    __shared__ float s_sc[kSc][kSc + 1];
    __shared__ unsigned short s_list[kSc * kSc];  // pixels that passed the quick test: ly * kSc + lx
    __shared__ int s_n;
    __shared__ float r_s[kFastThreads / 32];
    __shared__ int r_y[kFastThreads / 32], r_x[kFastThreads / 32];
    const int bx = blockIdx.x, by = blockIdx.y;
    const int y0 = (int)((long long)by * H / grid_y), y1 = (int)((long long)(by + 1) * H / grid_y);
    const int x0 = (int)((long long)bx * W / grid_x), x1 = (int)((long long)(bx + 1) * W / grid_x);
    float best_s = 0.f;
    int best_y = -1, best_x = -1;
    for (int sy0 = y0; sy0 < y1; sy0 += kSub)
        for (int sx0 = x0; sx0 < x1; sx0 += kSub) {
            const int sy1 = min(sy0 + kSub, y1), sx1 = min(sx0 + kSub, x1);
            const int niy = sy1 - sy0 + 8, nix = sx1 - sx0 + 8;  // staged rows and columns
            __syncthreads();  // the previous sub-tile's readers are done
            if (threadIdx.x == 0) s_n = 0;
            // flat indices over an n-wide area advance by kFastThreads: dq rows and dr columns
            {
                const int dq = kFastThreads / nix, dr = kFastThreads - dq * nix;
                int ly = threadIdx.x / nix, lx = threadIdx.x - ly * nix;
                while (ly < niy) {
                    const int gy = sy0 - 4 + ly, gx = sx0 - 4 + lx;
                    s_img[ly][lx] = (gy >= 0 && gy < H && gx >= 0 && gx < W) ? img[(size_t)gy * pitch + gx] : 0.f;
                    ly += dq;
                    lx += dr;
                    if (lx >= nix) {
                        lx -= nix;
                        ++ly;
                    }
                }
            }
            __syncthreads();
            {
                const int nsy = sy1 - sy0 + 2, nsx = sx1 - sx0 + 2;
                const int dq = kFastThreads / nsx, dr = kFastThreads - dq * nsx;
                int ly = threadIdx.x / nsx, lx = threadIdx.x - ly * nsx;
                while (ly < nsy) {
                    const int gy = sy0 - 1 + ly, gx = sx0 - 1 + lx;
                    if (!QUICK) {
                        float sc = 0.f;
                        if (gy >= 3 && gy < H - 3 && gx >= 3 && gx < W - 3) sc = fast_score(s_img, ly + 3, lx + 3, t);
                        if (sc > 0.f) s_list[atomicAdd(&s_n, 1)] = (unsigned short)(ly * kSc + lx);
                        s_sc[ly][lx] = sc;
                    } else if (gy >= 3 && gy < H - 3 && gx >= 3 && gx < W - 3) {
                        const int iy = ly + 3, ix = lx + 3;
                        const float c = s_img[iy][ix];
                        bool bright = true, dark = true;
#pragma unroll
                        for (int k = 0; k < 8; k += 2) {
                            const float a = s_img[iy + cdy(k)][ix + cdx(k)] - c;
                            const float b = s_img[iy + cdy(k + 8)][ix + cdx(k + 8)] - c;
                            // (NaN differences count as passing, as in the score's min and max)
                            bright = bright && !(a <= t && b <= t);
                            dark = dark && !(a >= -t && b >= -t);
                        }
                        if (bright || dark) s_list[atomicAdd(&s_n, 1)] = (unsigned short)(ly * kSc + lx);
                    }
                    if (QUICK) s_sc[ly][lx] = 0.f;
                    ly += dq;
                    lx += dr;
                    if (lx >= nsx) {
                        lx -= nsx;
                        ++ly;
                    }
                }
            }
            __syncthreads();
            const int nl = s_n;
            for (int i = threadIdx.x; i < (QUICK ? nl : 0); i += kFastThreads) {
                const int ly = s_list[i] / kSc, lx = s_list[i] - ly * kSc;
                const int iy = ly + 3, ix = lx + 3;  // staged position
                s_sc[ly][lx] = fast_score(s_img, iy, ix, t);
            }
            __syncthreads();
            for (int i = threadIdx.x; i < nl; i += kFastThreads) {
                const int ly = s_list[i] / kSc - 1, lx = s_list[i] - (ly + 1) * kSc - 1;
                const int gy = sy0 + ly, gx = sx0 + lx;
                if (ly < 0 || gy >= sy1 || lx < 0 || gx >= sx1) continue;  // the ring
                if (gy < margin || gy >= H - margin || gx < margin || gx >= W - margin) continue;
                const float v = s_sc[ly + 1][lx + 1];
                if (!(v > 0.f)) continue;
                bool keep = true;
#pragma unroll
                for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
                    for (int dx = -1; dx <= 1; ++dx) {
                        if (!dx && !dy) continue;
                        const int ny = gy + dy, nx = gx + dx;
                        if (ny < 0 || ny >= H || nx < 0 || nx >= W) continue;
                        const float u = s_sc[ly + 1 + dy][lx + 1 + dx];
                        const bool before = dy < 0 || (dy == 0 && dx < 0);
                        keep = keep && (before ? v > u : v >= u);
                    }
                if (keep && better(v, gy, gx, best_s, best_y, best_x)) {
                    best_s = v;
                    best_y = gy;
                    best_x = gx;
                }
            }
        }
    auto take = [&](float s, int y, int x) {
        if (better(s, y, x, best_s, best_y, best_x)) {
            best_s = s;
            best_y = y;
            best_x = x;
        }
    };
    for (int o = 16; o > 0; o >>= 1) {
        const float s = __shfl_down_sync(0xffffffffu, best_s, o);
        const int y = __shfl_down_sync(0xffffffffu, best_y, o), x = __shfl_down_sync(0xffffffffu, best_x, o);
        take(s, y, x);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        r_s[w] = best_s;
        r_y[w] = best_y;
        r_x[w] = best_x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < kFastThreads / 32; ++q) take(r_s[q], r_y[q], r_x[q]);
        const int b = by * grid_x + bx;
        points[2 * b] = best_x;
        points[2 * b + 1] = best_y;
        scores[b] = best_x >= 0 ? best_s : 0.f;
    }
}

}  // namespace

cudaError_t launch_fast_blocks(const float* img, int H, int W, size_t pitch, float t, int grid_y, int grid_x,
                               int margin, int32_t* points, float* scores, cudaStream_t st) {
    dim3 grid((unsigned)grid_x, (unsigned)grid_y);
    if (t > 0.f)
        k_fast_blocks<true><<<grid, kFastThreads, 0, st>>>(img, H, W, pitch, t, grid_y, grid_x, margin, points, scores);
    else
        k_fast_blocks<false><<<grid, kFastThreads, 0, st>>>(img, H, W, pitch, t, grid_y, grid_x, margin, points, scores);
    return cudaGetLastError();
}

}  // namespace sfoc

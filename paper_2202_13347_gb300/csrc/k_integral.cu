// Integral feature images (Eq. 14-16 of arXiv 2202.13347), exact.
//
// The two channel-summed planes s1 = sum_c g and s2 = sum_c g^2 of a cube
// are turned into exclusive prefix planes P[y][x] = sum over rows < y and
// columns < x, of size (H+1) x (W+1), so any window sum costs four lookups
// (Eq. 16).  Each pixel value is rounded once to a multiple of 2^-28 and
// the prefixes are integer sums in 64 bits, so every window sum is exact
// (its only error is the per-pixel rounding, at most 2^-29 per pixel) and
// no floating-point adds are needed: GB300's FP64 rate is a small fraction
// of its FP32 and integer rates.  The sums wrap modulo 2^64, which leaves
// window differences exact.  A non-finite value enters as 2^46; window
// sums of valid values stay below 2^45 (see internal.h), so a window sum at
// or above 2^45 marks a window with a non-finite value.
//
// Steps over tiles of 128 columns x 64 rows:
//   k_int_tilesums  per tile: column sums and row sums (reads s1, s2 once)
//   k_int_carry     running sums of those over the tiles above (left)
//   k_int_lines     P on the tile grid lines: a scan along each line
//   k_int_final     per tile: local 2-D prefix + the grid-line values
// HBM traffic is ~8 B/px read twice + 16 B/px written: 15 us of HBM time for a
// 2048 x 2048 cube.  A CTA takes one tile of one plane, a warp eight of its
// rows with four columns per lane: all eight rows' loads are in flight at once,
// a row's prefix is a lane's own three adds and one warp scan, and the eight
// warps meet once, at a table of their column sums.  (64 x 64 tiles in shared
// memory, where one thread per row and then per column adds 64 dependent
// entries, took twice the time; a single warp per tile, eight or four rows of
// loads in flight at a time, lost to them: the latency of 64 rows in a row.)
// 2048 x 2048, tilesums + carry + lines + final: 40 + 7 + 10 + 54 -> 15 + 6 + 9 + 30
// us; 512 x 512: 6 + 3 + 4 + 8 us.
#include <math.h>
#include <string.h>

#include "internal.h"

namespace sfoc {

namespace {

constexpr int kTR = 64, kTC = 128;  // tile rows and columns
constexpr int kIR = 8;              // rows per warp of the tile kernels
constexpr int kIntWarps = kTR / kIR;
typedef unsigned long long u64;

__device__ __forceinline__ u64 quant(float v) { return int_quant(v); }

struct IntLayout {
    int H, W, nty, ntx;
    u64* colsum;  // [2][nty][W]   column sums per tile row (then exclusive prefix over tile rows)
    u64* rowsum;  // [2][ntx][H]   row sums per tile column (then exclusive prefix over tile columns)
    u64* top;     // [2][nty][W+1] P[y0(ty)][x]
    u64* left;    // [2][ntx][H+1] P[y][x0(tx)]
};

IntLayout layout(int H, int W, void* scratch) {
    IntLayout L;
    L.H = H;
    L.W = W;
    L.nty = (H + kTR - 1) / kTR;
    L.ntx = (W + kTC - 1) / kTC;
    u64* p = static_cast<u64*>(scratch);
    L.colsum = p;
    p += 2 * (size_t)L.nty * W;
    L.rowsum = p;
    p += 2 * (size_t)L.ntx * H;
    L.top = p;
    p += 2 * (size_t)L.nty * (W + 1);
    L.left = p;
    return L;
}

// One cube's integral images: its sum planes, scratch layout and output.
struct IntJob {
    IntLayout L;
    const float* s1;
    const float* s2;
    size_t pitch;
    u64* P;
    size_t ipitch;
};

// CTAs of each of the four kernels for one cube
struct IntCtas {
    int tiles, carry, lines, fin;
};

IntCtas int_ctas(int H, int W) {
    const int nty = (H + kTR - 1) / kTR, ntx = (W + kTC - 1) / kTC;
    IntCtas c;
    c.tiles = 2 * ntx * nty;
    c.carry = (2 * W + 2 * H + 255) / 256;
    c.lines = 2 * nty + 2 * ntx;
    c.fin = c.tiles;
    return c;
}

// the job of this CTA (single: `one`, the CTA index as is) and the CTA's
// index within it (binary search of the prefix `begin` of n entries)
__device__ __forceinline__ const IntJob& int_job(const IntJob& one, const IntJob* jobs, const int* begin, int n,
                                                 int* local) {
    const int bid = blockIdx.x;
    if (!jobs) {
        *local = bid;
        return one;
    }
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (begin[mid] <= bid) lo = mid;
        else hi = mid - 1;
    }
    *local = bid - begin[lo];
    return jobs[lo];
}

// this warp's rows y .. y + kIR - 1 at the lane's columns x .. x + 3 (x a multiple
// of 4), zero past the image: rows are pitch (a multiple of 32) floats, so the
// load stays inside the row
__device__ __forceinline__ void int_rows(const float* __restrict__ s, size_t pitch, int y, int x, int H, int W,
                                         float4 (&f)[kIR]) {
#pragma unroll
    for (int r = 0; r < kIR; ++r) {
        f[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (x < W && y + r < H) f[r] = *reinterpret_cast<const float4*>(s + (size_t)(y + r) * pitch + x);
    }
}

// four columns' values rounded; zero past the image, whatever the row's padding holds
__device__ __forceinline__ void int_quant4(const float4& f, int x, int W, u64 (&q)[4]) {
    q[0] = x < W ? quant(f.x) : 0ull;
    q[1] = x + 1 < W ? quant(f.y) : 0ull;
    q[2] = x + 2 < W ? quant(f.z) : 0ull;
    q[3] = x + 3 < W ? quant(f.w) : 0ull;
}

// the tile of this CTA: plane *p, tile row *ty and column *tx
__device__ __forceinline__ void int_tile(const IntLayout& L, int local, int* p, int* ty, int* tx) {
    const int n = L.ntx * L.nty;
    *p = local >= n ? 1 : 0;
    local -= *p * n;
    *ty = local / L.ntx;
    *tx = local - *ty * L.ntx;
}

__global__ void __launch_bounds__(32 * kIntWarps)
    k_int_tilesums(const __grid_constant__ IntJob one, const IntJob* __restrict__ jobs, const int* __restrict__ begin,
                   int n_jobs) {
    __shared__ __align__(16) u64 s_col[kIntWarps][kTC];
    int local, p, ty, tx;
    const IntJob& J = int_job(one, jobs, begin, n_jobs, &local);
    const IntLayout& L = J.L;
    int_tile(L, local, &p, &ty, &tx);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, H = L.H, W = L.W;
    const int x0 = tx * kTC, x = x0 + 4 * lane, y0 = ty * kTR + w * kIR;
    float4 f[kIR];
    int_rows(p ? J.s2 : J.s1, J.pitch, y0, x, H, W, f);
    u64 col[4] = {0ull, 0ull, 0ull, 0ull}, rs[kIR];  // rs: this lane's part of each row's sum
#pragma unroll
    for (int r = 0; r < kIR; ++r) {
        u64 q[4];
        int_quant4(f[r], x, W, q);
#pragma unroll
        for (int c = 0; c < 4; ++c) col[c] += q[c];
        rs[r] = (q[0] + q[1]) + (q[2] + q[3]);
    }
    *reinterpret_cast<ulonglong2*>(&s_col[w][4 * lane]) = make_ulonglong2(col[0], col[1]);
    *reinterpret_cast<ulonglong2*>(&s_col[w][4 * lane + 2]) = make_ulonglong2(col[2], col[3]);
    // lanes exchange halves of the rows: lane l of each eight ends with its eight's
    // sum of row l, then the four eights are added
#pragma unroll
    for (int o = kIR / 2; o >= 1; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < kIR / 2; ++i)
            if (i < o) {
                const u64 give = up ? rs[i] : rs[i + o], keep = up ? rs[i + o] : rs[i];
                rs[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
    }
#pragma unroll
    for (int o = kIR; o < 32; o <<= 1) rs[0] += __shfl_xor_sync(0xffffffffu, rs[0], o);
    if (lane < kIR && y0 + lane < H) L.rowsum[((size_t)p * L.ntx + tx) * H + y0 + lane] = rs[0];
    __syncthreads();
    const int t = threadIdx.x;
    if (t < kTC && x0 + t < W) {
        u64 a = 0;
#pragma unroll
        for (int k = 0; k < kIntWarps; ++k) a += s_col[k][t];
        L.colsum[((size_t)p * L.nty + ty) * W + x0 + t] = a;
    }
}

// Exclusive running sums over tile rows (per column) and tile columns (per row).
__global__ void k_int_carry(const __grid_constant__ IntJob one, const IntJob* __restrict__ jobs,
                            const int* __restrict__ begin, int n_jobs) {
    int local;
    const IntJob& J = int_job(one, jobs, begin, n_jobs, &local);
    const IntLayout& L = J.L;
    size_t i = local * (size_t)blockDim.x + threadIdx.x;
    size_t ncol = 2 * (size_t)L.W, nrow = 2 * (size_t)L.H;
    // a line's values in groups of 8 loaded before any of them is replaced,
    // so the loads of a group overlap (one memory latency per group)
    auto carry = [](u64* __restrict__ base, size_t stride, int n) {
        u64 run = 0;
        for (int t0 = 0; t0 < n; t0 += 8) {
            u64 v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = t0 + k < n ? base[(size_t)(t0 + k) * stride] : 0ull;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (t0 + k < n) {
                    base[(size_t)(t0 + k) * stride] = run;
                    run += v[k];
                }
        }
    };
    if (i < ncol) {
        const int p = (int)(i / L.W), x = (int)(i % L.W);
        carry(&L.colsum[(size_t)p * L.nty * L.W + x], (size_t)L.W, L.nty);
    } else if (i < ncol + nrow) {
        i -= ncol;
        const int p = (int)(i / L.H), y = (int)(i % L.H);
        carry(&L.rowsum[(size_t)p * L.ntx * L.H + y], (size_t)L.H, L.ntx);
    }
}

// Block-wide exclusive scan of n values: out[0] = 0, out[k] = sum in[0..k-1].
__device__ void block_scan_excl(const u64* in, u64* out, int n) {
    __shared__ u64 warp_tot[32];
    __shared__ u64 carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int base = 0; base < n + 1; base += blockDim.x) {
        int k = base + threadIdx.x;      // out index
        u64 v = (k >= 1 && k - 1 < n) ? in[k - 1] : 0ull;
        // inclusive warp scan
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            u64 u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        if (lane == 31) warp_tot[wid] = v;
        __syncthreads();
        if (wid == 0) {
            u64 w = lane < nw ? warp_tot[lane] : 0ull;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                u64 u = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += u;
            }
            if (lane < nw) warp_tot[lane] = w;  // inclusive over warps
        }
        __syncthreads();
        u64 off = carry + (wid > 0 ? warp_tot[wid - 1] : 0ull);
        if (k <= n) out[k] = v + off;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = off + v;
        __syncthreads();
    }
}

// blocks [0, 2*nty): horizontal lines; [2*nty, 2*nty + 2*ntx): vertical lines
__global__ void __launch_bounds__(256) k_int_lines(const __grid_constant__ IntJob one, const IntJob* __restrict__ jobs,
                                                    const int* __restrict__ begin, int n_jobs) {
    int b;
    const IntJob& J = int_job(one, jobs, begin, n_jobs, &b);
    const IntLayout& L = J.L;
    if (b < 2 * L.nty) {
        int p = b / L.nty, ty = b % L.nty;
        block_scan_excl(&L.colsum[((size_t)p * L.nty + ty) * L.W], &L.top[((size_t)p * L.nty + ty) * (L.W + 1)], L.W);
    } else {
        b -= 2 * L.nty;
        int p = b / L.ntx, tx = b % L.ntx;
        block_scan_excl(&L.rowsum[((size_t)p * L.ntx + tx) * L.H], &L.left[((size_t)p * L.ntx + tx) * (L.H + 1)], L.H);
    }
}

__global__ void __launch_bounds__(32 * kIntWarps, 2)
    k_int_final(const __grid_constant__ IntJob one, const IntJob* __restrict__ jobs, const int* __restrict__ begin,
                int n_jobs) {
    __shared__ __align__(16) u64 s_col[kIntWarps][kTC];
    __shared__ __align__(16) u64 s_row[kIntWarps][2][kTC];
    int local, p, ty, tx;
    const IntJob& J = int_job(one, jobs, begin, n_jobs, &local);
    const IntLayout& L = J.L;
    int_tile(L, local, &p, &ty, &tx);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, H = L.H, W = L.W;
    const size_t ipitch = J.ipitch;
    u64* const Pp = J.P + (size_t)p * (H + 1) * ipitch;
    const u64* const top = &L.top[((size_t)p * L.nty + ty) * (W + 1)];
    const u64* const left = &L.left[((size_t)p * L.ntx + tx) * (H + 1)];
    const int x0 = tx * kTC, x = x0 + 4 * lane, y0 = ty * kTR + w * kIR;
    float4 f[kIR];
    int_rows(p ? J.s2 : J.s1, J.pitch, y0, x, H, W, f);
    // run[c]: P at column x + c down to the current row, less the line left of the
    // tile; it starts with the line above the tile
    const u64 corner = top[x0];
    u64 run[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) run[c] = (x + c < W ? top[x + c + 1] : 0ull) - corner;
    const u64 lft = lane < kIR && y0 + lane < H ? left[y0 + lane + 1] : 0ull;
    u64 pre[kIR][4], ex[kIR];  // the tile rows' prefixes
#pragma unroll
    for (int r = 0; r < kIR; ++r) {
        int_quant4(f[r], x, W, pre[r]);
        pre[r][1] += pre[r][0];
        pre[r][2] += pre[r][1];
        pre[r][3] += pre[r][2];
        ex[r] = pre[r][3];
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int r = 0; r < kIR; ++r) {
            const u64 v = __shfl_up_sync(0xffffffffu, ex[r], o);
            ex[r] += lane >= o ? v : 0ull;
        }
    u64 col[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
    for (int r = 0; r < kIR; ++r) {
        const u64 before = ex[r] - pre[r][3];  // the lanes to the left
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            pre[r][c] += before;
            col[c] += pre[r][c];
        }
    }
    *reinterpret_cast<ulonglong2*>(&s_col[w][4 * lane]) = make_ulonglong2(col[0], col[1]);
    *reinterpret_cast<ulonglong2*>(&s_col[w][4 * lane + 2]) = make_ulonglong2(col[2], col[3]);
    __syncthreads();
    for (int k = 0; k < w; ++k) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(&s_col[k][4 * lane]);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(&s_col[k][4 * lane + 2]);
        run[0] += a.x;
        run[1] += a.y;
        run[2] += b.x;
        run[3] += b.y;
    }
    u64 (*row)[kTC] = s_row[w];
#pragma unroll
    for (int r = 0; r < kIR; ++r) {
        const int y = y0 + r;
        const u64 l = __shfl_sync(0xffffffffu, lft, r);
#pragma unroll
        for (int c = 0; c < 4; ++c) run[c] += pre[r][c];
        // through shared memory, so that a store instruction writes 32 adjacent
        // entries (rows of W + 1 entries keep no wider alignment); two rows
        // alternate, so one warp barrier orders each
        u64* const buf = row[r & 1];
        *reinterpret_cast<ulonglong2*>(buf + 4 * lane) = make_ulonglong2(run[0] + l, run[1] + l);
        *reinterpret_cast<ulonglong2*>(buf + 4 * lane + 2) = make_ulonglong2(run[2] + l, run[3] + l);
        __syncwarp();
        u64* const out = Pp + (size_t)(y + 1) * ipitch + x0 + 1;
        if (y < H)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (x0 + 32 * c + lane < W) out[32 * c + lane] = buf[32 * c + lane];
    }
    // zero first row / column
    if (ty == 0 && w == 0)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (x0 + 32 * c + lane < W) Pp[x0 + 32 * c + lane + 1] = 0;
    if (tx == 0 && lane < kIR && y0 + lane < H) Pp[(size_t)(y0 + lane + 1) * ipitch] = 0;
    if (tx == 0 && ty == 0 && threadIdx.x == 0) Pp[0] = 0;
}

// ---- FP64 export: the prefix planes as doubles, NaN where the prefix
// rectangle holds a non-finite value (counted here, outside the hot path)
__global__ void k_nf_rows(const float* __restrict__ s1, const float* __restrict__ s2, size_t pitch, int H, int W,
                          int* __restrict__ C) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 2 * H) return;
    const int p = i / H, y = i - p * H;
    const float* s = (p ? s2 : s1) + (size_t)y * pitch;
    int* row = C + ((size_t)p * (H + 1) + y + 1) * (W + 1);
    int run = 0;
    row[0] = 0;
    for (int x = 0; x < W; ++x) {
        run += isfinite(s[x]) ? 0 : 1;
        row[x + 1] = run;
    }
}

__global__ void k_nf_cols(int H, int W, int* __restrict__ C) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 2 * (W + 1)) return;
    const int p = i / (W + 1), x = i - p * (W + 1);
    int* c = C + (size_t)p * (H + 1) * (W + 1) + x;
    c[0] = 0;
    int run = 0;
    for (int y = 1; y <= H; ++y) {
        run += c[(size_t)y * (W + 1)];
        c[(size_t)y * (W + 1)] = run;
    }
}

__global__ void k_int_to_f64(const u64* __restrict__ P, size_t ipitch, const int* __restrict__ C, int H, int W,
                             double* __restrict__ out) {
    const size_t n = 2 * (size_t)(H + 1) * (W + 1);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t pr = i / (W + 1);
        const int x = (int)(i - pr * (W + 1));
        const double v = (double)(long long)P[pr * ipitch + x] * (1.0 / kIntScale);
        out[i] = C[i] ? NAN : v;
    }
}

}  // namespace

size_t integral_export_scratch_bytes(int H, int W) { return sizeof(int) * 2 * (size_t)(H + 1) * (W + 1); }

cudaError_t launch_integral_export(const Cube& c, void* scratch, double* out, cudaStream_t st) {
    int* C = static_cast<int*>(scratch);
    k_nf_rows<<<(2 * c.H + 127) / 128, 128, 0, st>>>(c.s1, c.s2, c.pitch, c.H, c.W, C);
    k_nf_cols<<<(2 * (c.W + 1) + 127) / 128, 128, 0, st>>>(c.H, c.W, C);
    k_int_to_f64<<<8 * device_sms(), 256, 0, st>>>(c.integ, c.ipitch, C, c.H, c.W, out);
    return cudaGetLastError();
}

size_t integral_scratch_bytes(int H, int W) {
    size_t nty = (H + kTR - 1) / kTR, ntx = (W + kTC - 1) / kTC;
    return sizeof(u64) * (2 * nty * W + 2 * ntx * H + 2 * nty * (W + 1) + 2 * ntx * (H + 1));
}

namespace {

IntJob int_job_of(const Cube& c, void* scratch) {
    IntJob j;
    j.L = layout(c.H, c.W, scratch);
    j.s1 = c.s1;
    j.s2 = c.s2;
    j.pitch = c.pitch;
    j.P = c.integ;
    j.ipitch = c.ipitch;
    return j;
}

}  // namespace

cudaError_t launch_integral(const Cube& c, void* scratch, cudaStream_t st, int* launches) {
    const IntJob one = int_job_of(c, scratch);
    const IntCtas n = int_ctas(c.H, c.W);
    k_int_tilesums<<<n.tiles, 32 * kIntWarps, 0, st>>>(one, nullptr, nullptr, 0);
    k_int_carry<<<n.carry, 256, 0, st>>>(one, nullptr, nullptr, 0);
    k_int_lines<<<n.lines, 256, 0, st>>>(one, nullptr, nullptr, 0);
    k_int_final<<<n.fin, 32 * kIntWarps, 0, st>>>(one, nullptr, nullptr, 0);
    if (launches) *launches += 4;
    return cudaGetLastError();
}

// Batched form.  The table blob holds n IntJob entries and four prefix
// arrays (n + 1 ints each: tiles, carry, lines, final CTAs), in that order.
size_t integral_batch_blob_bytes(int n) {
    return ((sizeof(IntJob) * (size_t)n + 15) / 16) * 16 + 4 * sizeof(int) * (size_t)(n + 1);
}

void integral_batch_blob(const Cube* const* cubes, int n, char* scratch, void* blob, int* ctas4) {
    IntJob* jobs = static_cast<IntJob*>(blob);
    int* pre = reinterpret_cast<int*>(static_cast<char*>(blob) + ((sizeof(IntJob) * (size_t)n + 15) / 16) * 16);
    int acc[4] = {0, 0, 0, 0};
    for (int i = 0; i < n; ++i) {
        const Cube& c = *cubes[i];
        jobs[i] = int_job_of(c, scratch);
        scratch += (integral_scratch_bytes(c.H, c.W) + 255) / 256 * 256;
        const IntCtas k = int_ctas(c.H, c.W);
        const int v[4] = {k.tiles, k.carry, k.lines, k.fin};
        for (int q = 0; q < 4; ++q) {
            pre[q * (n + 1) + i] = acc[q];
            acc[q] += v[q];
        }
    }
    for (int q = 0; q < 4; ++q) {
        pre[q * (n + 1) + n] = acc[q];
        ctas4[q] = acc[q];
    }
}

size_t integral_batch_scratch_bytes(const Cube* const* cubes, int n) {
    size_t b = 0;
    for (int i = 0; i < n; ++i) b += (integral_scratch_bytes(cubes[i]->H, cubes[i]->W) + 255) / 256 * 256;
    return b;
}

cudaError_t launch_integral_batch(const void* d_blob, int n, const int* ctas4, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const IntJob* jobs = static_cast<const IntJob*>(d_blob);
    const int* pre =
        reinterpret_cast<const int*>(static_cast<const char*>(d_blob) + ((sizeof(IntJob) * (size_t)n + 15) / 16) * 16);
    IntJob none;
    memset(&none, 0, sizeof(none));
    k_int_tilesums<<<ctas4[0], 32 * kIntWarps, 0, st>>>(none, jobs, pre, n);
    k_int_carry<<<ctas4[1], 256, 0, st>>>(none, jobs, pre + (n + 1), n);
    k_int_lines<<<ctas4[2], 256, 0, st>>>(none, jobs, pre + 2 * (n + 1), n);
    k_int_final<<<ctas4[3], 32 * kIntWarps, 0, st>>>(none, jobs, pre + 3 * (n + 1), n);
    return cudaGetLastError();
}

}  // namespace sfoc

// NCC assembly, peak picking and sub-pixel refinement (Eq. 9, 12, 16 of
// arXiv 2202.13347; Sec. 3.2.2 takes the most similar position as the CP).
//
// k_template_stats  per point (one CTA): bounds check, then R_T and R_TT
//                   (Eq. 12) as sums of the sensed cube's channel-summed
//                   planes over the template, each pixel rounded to 2^-28
//                   units exactly as the integral images round it and added
//                   in 64-bit integers: the same exact values a lookup in
//                   integral images of the sensed cube would give, without
//                   building them.
// k_ncc_argmax      per point (one CTA): for every offset, R_S and R_SS from
//                   the reference integral images (4 lookups each, exact
//                   64-bit fixed point); the two steps that cancel are taken
//                   in exact 96-bit integers: mnz R_SS - R_S^2 (the
//                   variance times mnz) and, for the uncentred correlation
//                   forms, R_S R_T (the mean correction of the numerator);
//                   each is converted to FP32 (two roundings, relative error
//                   below 2^-23) and scaled by 2^-56 / mnz in FP32 (two more, the
//                   factor's and the product's), then NCC = num / sqrt(vS vT) in
//                   FP32; a warp-shuffle argmax with the (NCC desc, dy
//                   asc, dx asc) order and a 3-point parabola per axis.  No
//                   FP64 per offset: GB300 runs it at a small fraction of its
//                   FP32 rate, and the integer products cost a few 32-bit
//                   multiply-adds.
#include <math.h>
#include <string.h>

#include "internal.h"

namespace sfoc {

namespace {

typedef unsigned long long u64;

// A non-negative integer below 2^96 in 32-bit words.  Window sums in 2^-28 units
// stay below 2^45 in size and mnz below 2^19, so the exact products of the NCC fit
// it and take a handful of 32 x 32-bit multiply-adds (as 128-bit integers they
// took twice the instructions).
struct U96 {
    unsigned w0, w1, w2;
};

// a b, both below 2^45
__device__ __forceinline__ U96 mul96(u64 a, u64 b) {
    const unsigned al = (unsigned)a, ah = (unsigned)(a >> 32), bl = (unsigned)b, bh = (unsigned)(b >> 32);
    const u64 t0 = (u64)al * bl;
    const u64 t1 = (u64)al * bh + (u64)ah * bl + (t0 >> 32);  // below 2^47
    return {(unsigned)t0, (unsigned)t1, ah * bh + (unsigned)(t1 >> 32)};
}

// to FP32 from its first two words that count (two roundings, relative error below
// 2^-23; what a third word adds is below 2^-32 of it).  32-bit conversions: the
// 64-bit ones run on the FP64 pipe, 64 clocks a warp each.
__device__ __forceinline__ float u96_to_float(const U96& v) {
    const unsigned hi = v.w2 ? v.w2 : v.w1, lo = v.w2 ? v.w1 : v.w0;
    const float f = fmaf(__uint2float_rn(hi), 4294967296.f, __uint2float_rn(lo));
    return v.w2 ? f * 4294967296.f : f;
}

// Threads per point and loads in flight per thread: the two planes come from L2
// and a template is only m ceil(m / 32) warp loads of each, so a point's time is
// the number of dependent rounds of them: 128 threads with 4 loads took 36 us for
// 1000 points of m = 81, these 21 us (100 points of m = 41: 7 us).
constexpr int kStatThreads = 256, kStatLoads = 8;

__global__ void __launch_bounds__(kStatThreads)
    k_template_stats(const __grid_constant__ MatchJob one, const MatchJob* __restrict__ jobs,
                     const int2* __restrict__ items) {
    __shared__ u64 s_acc[kStatThreads / 32][2];
    int k;
    const MatchJob& J = item_job(one, jobs, items, blockIdx.x, &k);
    const float* __restrict__ s1 = J.ss1;
    const float* __restrict__ s2 = J.ss2;
    const size_t pitch = J.spitch;
    const int Hs = J.Hs, Ws = J.Ws, Hr = J.Hr, Wr = J.Wr, m = J.m, R = J.R, z = J.z;
    const int32_t* __restrict__ pts = J.pts;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int h = template_half(m);
    const int px = pts[2 * k], py = pts[2 * k + 1];
    const int ty0 = py - h, tx0 = px - h;
    const bool ok = ty0 >= 0 && tx0 >= 0 && ty0 + m <= Hs && tx0 + m <= Ws && ty0 - R >= 0 && tx0 - R >= 0 &&
                    ty0 + m + R <= Hr && tx0 + m + R <= Wr;
    u64 a1 = 0, a2 = 0;  // modulo 2^64, like the integral images
    if (ok) {
        // (row, column block) tasks of the template taken kStatLoads at a time per
        // warp, so that many loads are in flight before the first sum needs one
        const int ncol = (m + 31) >> 5;          // column blocks of 32 per row, at most 4 (m <= 128)
        const int ntask = m * ncol;
        const float inv = 1.f / (float)ncol;     // t / ncol is at least 1/8 from an integer after the + 1/2
        constexpr int kWarps = kStatThreads / 32;
        for (int t0 = warp; t0 < ntask; t0 += kStatLoads * kWarps) {
            float v1[kStatLoads], v2[kStatLoads];
#pragma unroll
            for (int u = 0; u < kStatLoads; ++u) {
                const int t = t0 + u * kWarps;
                const int r = (int)(((float)t + 0.5f) * inv), c = (t - r * ncol) * 32 + lane;
                const bool in = t < ntask && c < m;
                const size_t at = (size_t)(ty0 + (in ? r : 0)) * pitch + tx0 + (in ? c : 0);
                v1[u] = in ? s1[at] : 0.f;
                v2[u] = in ? s2[at] : 0.f;
            }
            // (a zero adds nothing)
#pragma unroll
            for (int u = 0; u < kStatLoads; ++u) {
                a1 += int_quant(v1[u]);
                a2 += int_quant(v2[u]);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a1 += __shfl_down_sync(0xffffffffu, a1, o);
        a2 += __shfl_down_sync(0xffffffffu, a2, o);
    }
    if (lane == 0) {
        s_acc[warp][0] = a1;
        s_acc[warp][1] = a2;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    PointStat s;
    s.rt = 0;
    s.tmean = s.vT = 0.f;
    if (!ok) {
        s.status = SFOC_PT_OUT_OF_BOUNDS;
    } else {
        u64 t1 = 0, t2 = 0;
        for (int w = 0; w < kStatThreads / 32; ++w) {
            t1 += s_acc[w][0];
            t2 += s_acc[w][1];
        }
        const long long rt = (long long)t1, rtt = (long long)t2;
        const double N = (double)m * m * z;
        if (rt >= kIntNonFiniteMin || rtt >= kIntNonFiniteMin) {
            s.status = SFOC_PT_NAN;
        } else {
            const double RT = int_units_to_double(rt), RTT = int_units_to_double(rtt);
            const double vT = RTT - RT * RT / N;
            s.rt = rt;
            s.vT = (float)vT;
            s.tmean = (float)(RT / N);
            s.status = vT <= 1e-6 * N ? SFOC_PT_FLAT_TEMPLATE : SFOC_PT_OK;
        }
    }
    J.stats[k] = s;
}

// argmax key: larger value wins, ties go to the smaller index
__device__ __forceinline__ bool better(float v, int i, float bv, int bi) {
    return v > bv || (v == bv && i < bi);
}

// What bounds the kernel: the lookups (64 B an offset from L2, little locality in
// L1) and ~80 instructions an offset.  Nothing of it may touch the FP64 pipe, which
// a warp's instruction holds for 64 clocks: what a point's warps all need in FP64
// is in its PointStat, or in the job.  Five CTAs per SM: more spill, fewer hide less
// of the lookups' latency (R = 40: 102 us, with four 126, with six 115; several
// offsets' lookups in flight per thread were slower too, 147 and 155).  With FP64
// in every warp, 128-bit products and the map in shared memory: 41 -> 31 us for
// 1000 points of R = 20, 146 -> 102 for 2000 of R = 40, 80 -> 65 for 400 of R = 60,
// 41 -> 25 for 2000 of R = 10.
constexpr int kNccThreads = 256;

__global__ void __launch_bounds__(kNccThreads, 5)
    k_ncc_argmax(const __grid_constant__ MatchJob one, const MatchJob* __restrict__ jobs,
                 const int2* __restrict__ items) {
    __shared__ float s_bv[kNccThreads / 32];
    __shared__ int s_bi[kNccThreads / 32];
    __shared__ int s_nan;
    int k;
    const MatchJob& J = item_job(one, jobs, items, blockIdx.x, &k);
    const u64* __restrict__ Pr = J.rint;
    const int Hr = J.Hr, m = J.m, R = J.R, centered = J.centered;
    const size_t ipr = J.ripitch;
    const int32_t* __restrict__ pts = J.pts;
    float* __restrict__ out_maps = J.out_maps;
    fastncc_result* __restrict__ out = J.out;
    const int P1 = 2 * R + 1, P = P1 * P1;
    const PointStat st = J.stats[k];
    if (threadIdx.x == 0) s_nan = 0;
    fastncc_result res;
    res.dx = res.dy = 0;
    res.ncc = 0.f;
    res.sub_dx = res.sub_dy = 0.f;
    res.status = st.status;
    if (st.status != SFOC_PT_OK) {
        if (out_maps)
            for (int i = threadIdx.x; i < P; i += blockDim.x) out_maps[(size_t)k * P + i] = 0.f;
        if (threadIdx.x == 0) out[k] = res;
        return;
    }
    __syncthreads();
    const unsigned Ni = (unsigned)(m * m * J.z);
    const float flat = J.flat, sc = J.sc, vTf = st.vT;
    const long long rt = st.rt;
    const u64 rta = (u64)(rt < 0 ? -rt : rt);
    const int h = template_half(m);
    const int ty0 = pts[2 * k + 1] - h, tx0 = pts[2 * k] - h;
    const u64* P1p = Pr;
    const size_t plane = (size_t)(Hr + 1) * ipr;
    // each numerator is replaced by its NCC: the peak's neighbours are read back
    // from there (a copy in shared memory kept CTAs out at large R)
    float* const nk = J.maps + (size_t)k * P;
    float bv = -INFINITY;
    int bi = 0x7fffffff;
    int has_nan = 0;
    // (i + 1/2) / P1 is at least 1 / (2 P1) from an integer, P1 <= 127: far more
    // than its two roundings
    const float inv = 1.f / (float)P1;
    const size_t dn = (size_t)m * ipr;
    for (int i = threadIdx.x; i < P; i += kNccThreads) {
        const int iy = (int)(((float)i + 0.5f) * inv), ix = i - iy * P1;
        const u64* a = P1p + (size_t)(ty0 + iy - R) * ipr + (tx0 + ix - R);
        const u64* b = a + plane;
        // window sums (Eq. 16) in 2^-28 units; exact (the planes wrap modulo 2^64)
        const long long rs = (long long)(a[dn + m] - a[m] - a[dn] + a[0]);
        const long long rss = (long long)(b[dn + m] - b[m] - b[dn] + b[0]);
        const float n32 = nk[i];
        float v;
        if (rs >= kIntNonFiniteMin || rss >= kIntNonFiniteMin || n32 != n32) {
            v = NAN;
        } else {
            // mnz R_SS - R_S^2, exact (units 2^-56); negative only through the
            // per-pixel rounding of a flat window
            const u64 rsa = (u64)(rs < 0 ? -rs : rs);
            const u64 x = (u64)Ni * (unsigned)rss + ((u64)(Ni * (unsigned)((u64)rss >> 32)) << 32);
            const U96 q = mul96(rsa, rsa);
            const u64 xl = x << 28, ql = (u64)q.w1 << 32 | q.w0, dl = xl - ql;
            const int d2 = (int)((unsigned)(x >> 36) - q.w2 - (xl < ql ? 1u : 0u));
            const float vS = d2 >= 0 ? u96_to_float({(unsigned)dl, (unsigned)(dl >> 32), (unsigned)d2}) * sc : 0.f;
            float nm = n32;
            if (!centered) {
                const float pf = u96_to_float(mul96(rsa, rta));  // |R_S R_T|, exact
                nm = fmaf((rs < 0) != (rt < 0) ? pf : -pf, sc, n32);
            }
            v = vS <= flat ? 0.f : nm / sqrtf(vS * vTf);
        }
        nk[i] = v;
        if (out_maps) out_maps[(size_t)k * P + i] = v;
        if (v != v) { has_nan = 1; continue; }
        if (better(v, i, bv, bi)) { bv = v; bi = i; }
    }
    // warp argmax
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        float ov = __shfl_down_sync(full, bv, o);
        int oi = __shfl_down_sync(full, bi, o);
        if (better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
    }
    has_nan = __any_sync(full, has_nan);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        s_bv[wid] = bv;
        s_bi[wid] = bi;
        if (has_nan) atomicOr(&s_nan, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        bv = s_bv[0];
        bi = s_bi[0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            if (better(s_bv[w], s_bi[w], bv, bi)) { bv = s_bv[w]; bi = s_bi[w]; }
        if (bi == 0x7fffffff) {  // every score NaN
            res.status = SFOC_PT_NAN;
        } else {
            int iy = bi / P1, ix = bi - iy * P1;
            res.dy = iy - R;
            res.dx = ix - R;
            res.ncc = (float)bv;
            bool edge = false;
            double ddx = 0.0, ddy = 0.0;
            auto parab = [](double cm, double c0, double cp) {  // from the FP32 map values
                double den = cm - 2.0 * c0 + cp;
                if (!(den < 0.0)) return 0.0;
                double d = (cm - cp) / (2.0 * den);
                return d > 0.5 ? 0.5 : (d < -0.5 ? -0.5 : d);
            };
            if (ix > 0 && ix < P1 - 1) ddx = parab(nk[bi - 1], bv, nk[bi + 1]);
            else edge = true;
            if (iy > 0 && iy < P1 - 1) ddy = parab(nk[bi - P1], bv, nk[bi + P1]);
            else edge = true;
            if (ddx != ddx) ddx = 0.0;
            if (ddy != ddy) ddy = 0.0;
            res.sub_dx = (float)(res.dx + ddx);
            res.sub_dy = (float)(res.dy + ddy);
            res.status = s_nan ? SFOC_PT_NAN : (edge ? SFOC_PT_PEAK_ON_EDGE : SFOC_PT_OK);
        }
        out[k] = res;
    }
}

}  // namespace

cudaError_t launch_template_stats(const MatchJob& one, const ItemSet& is, cudaStream_t st) {
    const int n = is.items ? is.n : one.n;
    if (n <= 0) return cudaSuccess;
    k_template_stats<<<n, kStatThreads, 0, st>>>(one, is.jobs, is.items);
    return cudaGetLastError();
}

cudaError_t launch_ncc_argmax(const MatchJob& one, const ItemSet& is, cudaStream_t st) {
    const int n = is.items ? is.n : one.n;
    if (n <= 0) return cudaSuccess;
    k_ncc_argmax<<<n, kNccThreads, 0, st>>>(one, is.jobs, is.items);
    return cudaGetLastError();
}

MatchJob make_job(const Cube& ref, const Cube& sen, const int32_t* pts, int n, int m, int R, PointStat* stats,
                  float* maps, float* out_maps, fastncc_result* out) {
    MatchJob j;
    memset(&j, 0, sizeof(j));
    j.rf32 = ref.f32;
    j.rrm = ref.rm;
    j.rcm = ref.cm;
    j.rpl = ref.pl;
    j.rint = ref.integ;
    j.rpitch = ref.pitch;
    j.rplane = ref.pitch * (size_t)ref.H;
    j.ripitch = ref.ipitch;
    j.Hr = ref.H;
    j.Wr = ref.W;
    j.sf32 = sen.f32;
    j.ss1 = sen.s1;
    j.ss2 = sen.s2;
    j.srm = sen.rm;
    j.scm = sen.cm;
    j.spl = sen.pl;
    j.spitch = sen.pitch;
    j.splane = sen.pitch * (size_t)sen.H;
    j.Hs = sen.H;
    j.Ws = sen.W;
    j.z = ref.z;
    j.m = m;
    j.R = R;
    j.n = n;
    j.pts = pts;
    j.stats = stats;
    j.maps = maps;
    j.out_maps = out_maps;
    const double N = (double)m * m * ref.z;
    j.flat = (float)(1e-6 * N);
    j.sc = (float)(1.0 / (72057594037927936.0 * N));
    j.out = out;
    return j;
}

}  // namespace sfoc

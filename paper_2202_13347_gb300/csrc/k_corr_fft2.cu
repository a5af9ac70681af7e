// Correlation R_ST (Eq. 10 of arXiv 2202.13347) by the discrete Fourier
// transform, Eq. 13: per point and channel the window S_c and the zero-mean
// template T_c - mean(T) are zero-padded to L x L (L >= m + 2R, so the
// circular correlation equals the linear one at every offset in [0, 2R]),
// their spectra multiplied (one conjugated) and summed over the channels,
// and one inverse transform gives the numerator of Eq. 9 at every offset.
// FP32 throughout, from the F32 cube or the planes of the BF16 cube; one CTA
// per point.
//
// Scheme.  Channel c: z = S_c + i (T_c - mean) is transformed once; the
// spectra of the two real inputs follow from Z[k] and conj(Z[-k]):
//   X = (Z[k] + conj Z[-k]) / 2,  Y = (Z[k] - conj Z[-k]) / 2i,
// and X conj(Y) is summed over the channels.  The columns kx of the spectrum
// are taken in two halves, the even ones (q = 0) and the odd ones (q = 1):
// both are closed under kx -> -kx, a half of the L x L array is all that shared
// memory holds (which lets sides up to 224 fit, and four or two CTAs per SM at
// 96 and 160), and the half's first radix-2 step is the first step of the row
// transform anyway.  The channel sums of both halves live in tensor memory
// (up to 448 columns): in registers they left the transforms spilling.
//
// With Lh = L / 2 columns, PR = L / 8, PC = L / 16 a half of channel c is
//   A  rows: x = t + PR j (j < 8): the radix-2 step over x and x + Lh, the
//      4-point DFT over the other j, twiddle W_L^{t (2 k1 + q)};
//   B  rows: PR-point DFT over t: column k1 + 4 k2 (kx = 2 (k1 + 4 k2) + q);
//      columns >= Lh / 2 are stored conjugated, so that their column transform
//      gives conj Z[-k] at the index of Z[k];
//   C  columns: y = t + PC j (j < 16): 16-point DFT over j, twiddle W_L^{t k1};
//   D  columns: PC-point DFTs over t of a column and its partner, ky = k1 + 16 k2,
//      cross spectrum added to the sums.
// Columns 0 and Lh / 2 of the even half pair with themselves; their spectra go
// through shared memory and every thread adds one of their 2 L bins.
// Every step works in place on the shared array.  A and B of a row belong to
// one warp (rows y = w + PC i), so a half costs three block barriers.  A
// channel's halves follow one another (the second finds its rows in L2), and
// the next channel's rows are prefetched into L2 meanwhile.
// The inverse runs the same steps backwards: D and C over the sums, then the
// 2R + 1 wanted rows (Hermitian extension), whose halves add up in the map.
//
// What bounds it: the shared-memory pipe (64 % busy at L = 160; six 64-bit
// accesses per element, channel and pass) and the row loads' latency, at 2.3
// instructions per clock.  Per point of 2000 on a 2048 x 2048 pair, F32 (BF16)
// cubes: m = 81, R = 36 1.40 (1.43) us, R = 40 1.92 (2.05), m = 80, R = 60 2.90
// (3.04), m = 61, R = 16 0.47.  The forms these windows had before: the direct
// kernel 40, 52 and 112 us (F32), the band and Toeplitz tensor-core forms 2.32,
// 3.02 and 10.2 us (BF16), the 128-point transform 0.75 us.
#include <math.h>

#include <type_traits>

#include "internal.h"

namespace sfoc {

namespace {

// CTAs per SM (MINB) and row items whose loads a thread has in flight together
// (UA): more of them hide more of the loads' latency but spill where the
// side's CTAs share the register file.
template <int L>
struct FftShape {
    static constexpr int Lh = L / 2, PR = L / 8, PC = L / 16;
    static constexpr int NT = 32 * PC;        // threads: one warp per residue of the rows modulo PC
    static constexpr int NI = 2;              // column-pair items per thread
    static constexpr int MINB = L <= 96 ? 4 : L <= 160 ? 2 : 1;
    static constexpr int UA = L == 96 || L == 192 ? 2 : 1;
    // windows of this side are larger than the next smaller one
    static constexpr int LMIN = L - 31;
    static constexpr size_t smem = sizeof(float2) * ((size_t)L * Lh + 2 * 4 * PR + 16 * PC + 2 * L);
    // tensor-memory columns: 2 PC words per item, for both halves, one lane
    // quarter per warp modulo 4; MINB CTAs hold at most the SM's 512
    static constexpr int tm_half = ((NT / 32 + 3) / 4) * NI * 2 * PC;
    static constexpr int tm_cols = 2 * tm_half <= 128 ? 128 : 2 * tm_half <= 256 ? 256 : 512;
    static_assert(MINB * tm_cols <= 512, "tensor memory of an SM");
};

// exp(-2 pi i n / L) for an integer n: a quarter turn and a rest of at most an
// eighth turn either side, so that the angle's rounding stays below 2^-26
__device__ __forceinline__ float2 unit_root(int n, int L) {
    n %= L;
    const int quarter = (8 * n + L) / (2 * L);  // nearest quarter turn
    float s, c;
    sincospif((float)(4 * n - quarter * L) / (float)(2 * L), &s, &c);
    switch (quarter & 3) {
        case 0: return make_float2(c, -s);
        case 1: return make_float2(-s, -c);
        case 2: return make_float2(-c, s);
        default: return make_float2(s, c);
    }
}

// N (a multiple of 4) 32-bit words per lane to or from tensor memory at
// `addr`, in runs of 16, 8 and 4 columns; tm_wait_ld / tm_wait_st complete them
// for the warp.
__device__ __forceinline__ void tm_ld(uint32_t addr, float* v, int n) {
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    if (n == 16)
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(addr));
    else if (n == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "r"(addr));
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(addr));
}
__device__ __forceinline__ void tm_st(uint32_t addr, const float* v, int n) {
    const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
    if (n == 16)
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
                addr),
            "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
            "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
            : "memory");
    else if (n == 8)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(addr), "r"(r[0]),
                     "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                     : "memory");
    else
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r[0]), "r"(r[1]),
                     "r"(r[2]), "r"(r[3])
                     : "memory");
}
__device__ __forceinline__ void tm_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void tm_load(uint32_t addr, float2 (&v)[N]) {
    float* f = reinterpret_cast<float*>(v);
    constexpr int W = 2 * N;
    if constexpr (W >= 16) tm_ld(addr, f, 16);
    if constexpr (W & 8) tm_ld(addr + (W & 16), f + (W & 16), 8);
    if constexpr (W & 4) tm_ld(addr + (W & 24), f + (W & 24), 4);
}
template <int N>
__device__ __forceinline__ void tm_store(uint32_t addr, const float2 (&v)[N]) {
    const float* f = reinterpret_cast<const float*>(v);
    constexpr int W = 2 * N;
    if constexpr (W >= 16) tm_st(addr, f, 16);
    if constexpr (W & 8) tm_st(addr + (W & 16), f + (W & 16), 8);
    if constexpr (W & 4) tm_st(addr + (W & 24), f + (W & 24), 4);
}

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cmul_conj(float2 a, float2 b) {  // a conj(b)
    return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
template <int SIGN>
__device__ __forceinline__ float2 rot(float2 v) {  // SIGN i v
    return SIGN < 0 ? make_float2(v.y, -v.x) : make_float2(-v.y, v.x);
}

// cos(2 pi q / 16)
__device__ __forceinline__ constexpr float cos16(int q) {
    constexpr float c[16] = {1.f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f,
                             0.f, -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128674f,
                             -1.f, -0.92387953251128674f, -0.70710678118654752f, -0.38268343236508977f,
                             0.f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128674f};
    return c[q & 15];
}

// x exp(SIGN 2 pi i k / N), N a divisor of 16, k a constant after unrolling
template <int SIGN>
__device__ __forceinline__ float2 twiddle(float2 x, int k, int N) {
    const int q = (k * (16 / N)) & 15;
    if (q == 0) return x;
    if (q == 8) return make_float2(-x.x, -x.y);
    if (q == 4) return rot<SIGN>(x);
    if (q == 12) return rot<-SIGN>(x);
    const float c = cos16(q), s = SIGN * cos16(q + 12);
    return make_float2(fmaf(x.x, c, -x.y * s), fmaf(x.x, s, x.y * c));
}

// In-register N-point DFTs, sum_j v[j] exp(SIGN 2 pi i j k / N), natural order.
// 2, 3, 4, 5, 7 directly; 8 and 16 by Cooley-Tukey; 6, 10, 12, 14, 20, 24, 28
// by the prime-factor map (coprime factors, no twiddles).
template <int N, int SIGN>
struct Dft;

template <int N, int SIGN>
__device__ __forceinline__ void dft(float2 (&v)[N]) {
    Dft<N, SIGN>::run(v);
}

template <int SIGN>
struct Dft<2, SIGN> {
    __device__ __forceinline__ static void run(float2 (&v)[2]) {
        const float2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    }
};
template <int SIGN>
struct Dft<3, SIGN> {
    __device__ __forceinline__ static void run(float2 (&v)[3]) {
        constexpr float s3 = 0.86602540378443865f;
        const float2 p = cadd(v[1], v[2]);
        const float2 d = rot<SIGN>(csub(v[1], v[2]));
        const float2 m = make_float2(fmaf(-0.5f, p.x, v[0].x), fmaf(-0.5f, p.y, v[0].y));
        v[0] = cadd(v[0], p);
        v[1] = make_float2(fmaf(s3, d.x, m.x), fmaf(s3, d.y, m.y));
        v[2] = make_float2(fmaf(-s3, d.x, m.x), fmaf(-s3, d.y, m.y));
    }
};
template <int SIGN>
struct Dft<4, SIGN> {
    __device__ __forceinline__ static void run(float2 (&v)[4]) {
        const float2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = rot<SIGN>(csub(v[1], v[3]));
        v[0] = cadd(a, c);
        v[2] = csub(a, c);
        v[1] = cadd(b, d);
        v[3] = csub(b, d);
    }
};
// odd prime N: pairs v[j] +- v[N - j], the cosine and sine sums of Eq. DFT
template <int N, int SIGN>
struct DftOdd {
    __device__ __forceinline__ static constexpr float cs(int q, bool sine) {
        // cos and sin of 2 pi q / 5 and 2 pi q / 7, q = 0 .. (N - 1) / 2
        constexpr float c5[3] = {1.f, 0.30901699437494742f, -0.80901699437494742f};
        constexpr float s5[3] = {0.f, 0.95105651629515357f, 0.58778525229247313f};
        constexpr float c7[4] = {1.f, 0.62348980185873353f, -0.22252093395631440f, -0.90096886790241913f};
        constexpr float s7[4] = {0.f, 0.78183148246802981f, 0.97492791218182361f, 0.43388373911755812f};
        const int r = q % N, h = r <= N / 2 ? r : N - r;
        if (sine) return (r <= N / 2 ? 1.f : -1.f) * (N == 5 ? s5[h % 3] : s7[h % 4]);
        return N == 5 ? c5[h % 3] : c7[h % 4];
    }
    __device__ __forceinline__ static void run(float2 (&v)[N]) {
        constexpr int M = N / 2;
        float2 p[M], d[M];
#pragma unroll
        for (int j = 1; j <= M; ++j) {
            p[j - 1] = cadd(v[j], v[N - j]);
            d[j - 1] = rot<SIGN>(csub(v[j], v[N - j]));
        }
        const float2 x0 = v[0];
#pragma unroll
        for (int j = 0; j < M; ++j) v[0] = cadd(v[0], p[j]);
#pragma unroll
        for (int k = 1; k <= M; ++k) {
            float2 e = x0, o = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 1; j <= M; ++j) {
                const float c = cs(j * k, false), s = cs(j * k, true);
                e = make_float2(fmaf(c, p[j - 1].x, e.x), fmaf(c, p[j - 1].y, e.y));
                o = j == 1 ? make_float2(s * d[0].x, s * d[0].y)
                           : make_float2(fmaf(s, d[j - 1].x, o.x), fmaf(s, d[j - 1].y, o.y));
            }
            v[k] = cadd(e, o);
            v[N - k] = csub(e, o);
        }
    }
};
template <int SIGN>
struct Dft<5, SIGN> : DftOdd<5, SIGN> {};
template <int SIGN>
struct Dft<7, SIGN> : DftOdd<7, SIGN> {};

// N = N1 N2 dividing 16: n = N2 n1 + n2, k = k1 + N1 k2
template <int N1, int N2, int SIGN>
struct DftCT {
    static constexpr int N = N1 * N2;
    __device__ __forceinline__ static void run(float2 (&v)[N]) {
        float2 u[N2][N1];
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) {
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) u[n2][n1] = v[N2 * n1 + n2];
            dft<N1, SIGN>(u[n2]);
        }
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
            float2 w[N2];
#pragma unroll
            for (int n2 = 0; n2 < N2; ++n2) w[n2] = twiddle<SIGN>(u[n2][k1], n2 * k1, N);
            dft<N2, SIGN>(w);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) v[k1 + N1 * k2] = w[k2];
        }
    }
};
template <int SIGN>
struct Dft<8, SIGN> : DftCT<4, 2, SIGN> {};
template <int SIGN>
struct Dft<16, SIGN> : DftCT<4, 4, SIGN> {};

// N = N1 N2, coprime: n = (N2 n1 + N1 n2) mod N; k = k1 mod N1 and k2 mod N2
template <int N1, int N2, int SIGN>
struct DftPF {
    static constexpr int N = N1 * N2;
    __device__ __forceinline__ static void run(float2 (&v)[N]) {
        float2 u[N2][N1];
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) {
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) u[n2][n1] = v[(N2 * n1 + N1 * n2) % N];
            dft<N1, SIGN>(u[n2]);
        }
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
            float2 w[N2];
#pragma unroll
            for (int n2 = 0; n2 < N2; ++n2) w[n2] = u[n2][k1];
            dft<N2, SIGN>(w);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                // the k with k = k1 (mod N1) and k = k2 (mod N2)
                int k = k2;
#pragma unroll
                for (int q = 0; q < N1; ++q)
                    if ((k2 + q * N2) % N1 == k1) k = k2 + q * N2;
                v[k] = w[k2];
            }
        }
    }
};
template <int SIGN>
struct Dft<6, SIGN> : DftPF<3, 2, SIGN> {};
template <int SIGN>
struct Dft<10, SIGN> : DftPF<5, 2, SIGN> {};
template <int SIGN>
struct Dft<12, SIGN> : DftPF<3, 4, SIGN> {};
template <int SIGN>
struct Dft<14, SIGN> : DftPF<7, 2, SIGN> {};
template <int SIGN>
struct Dft<20, SIGN> : DftPF<5, 4, SIGN> {};
template <int SIGN>
struct Dft<24, SIGN> : DftPF<3, 8, SIGN> {};
template <int SIGN>
struct Dft<28, SIGN> : DftPF<7, 4, SIGN> {};

// acc += 4 X conj(Y) (the factor is in the final scale), a = Z[k], b = conj(Z[-k])
__device__ __forceinline__ void cross_add(float2& acc, float2 a, float2 b) {
    const float2 s = cadd(a, b), d = csub(a, b);
    acc.x = fmaf(s.x, d.y, acc.x);
    acc.x = fmaf(-s.y, d.x, acc.x);
    acc.y = fmaf(s.x, d.x, acc.y);
    acc.y = fmaf(s.y, d.y, acc.y);
}

__device__ __forceinline__ float widen(float v) { return v; }
__device__ __forceinline__ float widen(__nv_bfloat16 v) { return __bfloat162float(v); }

// Slot of column c in a row of the shared array (rows of L / 2 float2): the
// low four bits carry a swizzle by the 16-column block (bits 0-1) and by the
// row's index i = y / PC (bits 2-3), so that the accesses of steps A (fixed
// column of 4-blocks, along t), B (4 columns x 4 rows), C and D (16 columns of
// a row) each fall on distinct banks.
__device__ __forceinline__ constexpr int swz_c(int c) { return c ^ ((c >> 4) & 3); }
__device__ __forceinline__ constexpr int swz_i(int i) { return (i & 3) << 2; }

// The shared array by byte offset.  A row is a multiple of 128 bytes and the
// swizzle touches bits 3-6 of an offset, so a neighbour in the swizzle is one
// XOR of an immediate away and a neighbour in another 16-column block or row an
// immediate of the access itself.
__device__ __forceinline__ float2& z_at(int off) {
    extern __shared__ __align__(128) float2 fsm[];
    return *reinterpret_cast<float2*>(reinterpret_cast<char*>(fsm) + off);
}

// One point's window and template (top-left value of channel 0) and its map.
template <typename T>
struct FftItem {
    const T* S;
    const T* T0;
    size_t splane, tplane;  // elements per channel
    unsigned spitch, tpitch;
    int m, Lw, P1, nch;
    float tmean;
    float* out;
};

// Items: the points of `one` (items == nullptr) or (job, point) pairs of a
// batch; with a queue the CTAs take items from an atomic counter (points of
// uneven cost balance across the SMs), else item k goes to CTA k mod grid.
// T: the cube's element type, planar [z][H][pitch] for both.
template <int L, typename T>
__global__ void __launch_bounds__(FftShape<L>::NT, FftShape<L>::MINB)
    k_corr_fft2(const __grid_constant__ MatchJob one, const MatchJob* __restrict__ jobs,
               const int2* __restrict__ items, int n_items, int* __restrict__ queue) {
    using Sh = FftShape<L>;
    constexpr int Lh = Sh::Lh, PR = Sh::PR, PC = Sh::PC, NT = Sh::NT, NI = Sh::NI, ZP = Lh;
    constexpr int RI = 16;  // rows a warp owns
    extern __shared__ __align__(128) float2 fsm[];
    // L x ZP values at offset 0 (z_at), rows y = w + PC i
    constexpr int ZB = ZP * 8;          // bytes per row
    float2* twr = fsm + (size_t)L * ZP;  // [q][k1][t]: W_L^{t (2 k1 + q)}
    float2* twc = twr + 2 * 4 * PR;     // [k1][t]: W_L^{t k1}
    float2* ex = twc + 16 * PC;         // [2][L]: columns 0 and Lh / 2 of the even half
    __shared__ int s_item;
    __shared__ uint32_t s_tmem;
    __shared__ FftItem<T> s_it;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rw = warp;                // the warp's rows: y = rw + PC i

    // the channel sums: 2 PC words per item and lane, the warp's lane quarter
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(&s_tmem)),
                     "r"(Sh::tm_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int p = tid; p < 2 * 4 * PR; p += NT) {
        const int q = p / (4 * PR), k1 = (p / PR) & 3, t = p % PR;
        twr[p] = unit_root(t * (2 * k1 + q), L);
    }
    for (int p = tid; p < 16 * PC; p += NT) {
        twc[p] = unit_root((p / PC) * (p % PC), L);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const uint32_t tacc = tmem + ((uint32_t)(warp & 3) << 21) + (uint32_t)((warp >> 2) * NI * 2 * PC);

    bool clean = false;  // the item is taken again with non-finite values as zeros
    int kk = 0;
    for (int next = blockIdx.x;;) {
        if (!clean) {
            if (queue) {
                if (tid == 0) s_item = atomicAdd(queue, 1);
                __syncthreads();
                kk = s_item;
                __syncthreads();  // read by all before thread 0 takes the next one
            } else {
                kk = next;
                next += gridDim.x;
            }
        }
        if (kk >= n_items) break;
        int k;
        const MatchJob& J = item_job(one, jobs, items, kk, &k);
        const PointStat st = J.stats[k];
        if (st.status != SFOC_PT_OK) continue;  // uniform across the CTA (and never with `clean`)
        // the item's sizes and pointers, in shared memory: read again after each
        // barrier, they hold no registers across the transforms
        if (tid == 0) {
            const int m = J.m, R = J.R;
            const int h = template_half(m);
            const int ty0 = J.pts[2 * k + 1] - h, tx0 = J.pts[2 * k] - h;
            const T* S0;
            const T* T0;
            if constexpr (std::is_same<T, float>::value) {
                S0 = J.rf32;
                T0 = J.sf32;
            } else {
                S0 = J.rpl;
                T0 = J.spl;
            }
            s_it.S = S0 + (size_t)(ty0 - R) * J.rpitch + (tx0 - R);
            s_it.T0 = T0 + (size_t)ty0 * J.spitch + tx0;
            s_it.splane = J.rplane;
            s_it.tplane = J.splane;
            s_it.spitch = (unsigned)J.rpitch;
            s_it.tpitch = (unsigned)J.spitch;
            s_it.m = m;
            s_it.Lw = m + 2 * R;
            s_it.P1 = 2 * R + 1;
            s_it.nch = J.z;
            s_it.tmean = st.tmean;
            s_it.out = J.maps + (size_t)k * (2 * R + 1) * (2 * R + 1);
        }
        __syncthreads();
        bool again = false;

        {
            float2 zero[PC];
#pragma unroll
            for (int j = 0; j < PC; ++j) zero[j] = make_float2(0.f, 0.f);
#pragma unroll
            for (int r = 0; r < 2 * NI; ++r) tm_store(tacc + (r / NI) * Sh::tm_half + (r % NI) * 2 * PC, zero);
        }
        float2 self = make_float2(0.f, 0.f);  // bin tid of the even half's self-paired columns
        auto add_self = [&]() {
            if (tid < L) {
                const float2 a = ex[tid], p = ex[tid ? L - tid : 0];
                cross_add(self, a, make_float2(p.x, -p.y));
            } else if (tid < 2 * L) {
                const int ky = tid - L;
                const float2 b = ex[tid], p = ex[L + (ky ? L - ky : 0)];
                cross_add(self, make_float2(p.x, -p.y), b);
            }
        };
        // a channel's two halves one after the other: the second finds the rows in L2
#pragma unroll 1
        for (int cq = 0; cq < 2 * s_it.nch; ++cq) {
            const int c = cq >> 1, q = cq & 1;
            {
                // ---- A: rows, radix 2 and 4
                const T* const Sc = s_it.S + (size_t)c * s_it.splane;
                const T* const Tc = s_it.T0 + (size_t)c * s_it.tplane;
                const unsigned spitch = s_it.spitch, tpitch = s_it.tpitch;
                const int m = s_it.m, Lw = s_it.Lw;
                const float tmean = s_it.tmean;
                // rows of this warp below Lw
                const int rows = min(max((Lw - rw + PC - 1) / PC, 0), RI);
                // UA items at a time, every load of them in flight before the first
                // is used (the loads come from L2 or HBM).  Item (i, t) of a lane
                // advances by 32: DI rows and DT columns, one row more on a wrap.
                constexpr int DI = 32 / PR, DT = 32 % PR;
                int ai = lane / PR, at = lane - ai * PR;
                const T* sp = Sc + (size_t)(rw + PC * ai) * spitch + at;
                const T* tp = Tc + (size_t)(rw + PC * ai) * tpitch + at;
                const size_t s1 = (size_t)(PC * DI) * spitch + DT, s2 = (size_t)PC * spitch - PR;
                const size_t t1 = (size_t)(PC * DI) * tpitch + DT, t2 = (size_t)PC * tpitch - PR;
                for (int it0 = 0; it0 < rows * PR; it0 += 32 * Sh::UA) {
                    float2 z[Sh::UA][8];
                    int offs[Sh::UA], ts[Sh::UA];
#pragma unroll
                    for (int u = 0; u < Sh::UA; ++u) {
                        const int y = rw + PC * ai;
                        const bool on = ai < rows;
                        const T* const sq = on ? sp : Sc;               // (a lane past the rows reads, and drops, row 0)
                        const int lw = Lw - at;                         // window columns left of x = t
                        const int mt = on && y < m ? m - at : 0;        // template columns
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            z[u][j].x = (PR * j + PR - 1 < Sh::LMIN || PR * j < lw) ? widen(sq[PR * j]) : 0.f;
                        // (rows below the template skip its loads where several CTAs share
                        // the SM; with one, the branch costs the loads' overlap more)
                        if (Sh::MINB == 1 || __any_sync(0xffffffffu, mt > 0)) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) z[u][j].y = PR * j < mt ? widen(tp[PR * j]) - tmean : 0.f;
                        } else {  // rows below the template
#pragma unroll
                            for (int j = 0; j < 8; ++j) z[u][j].y = 0.f;
                        }
                        offs[u] = on ? y * ZB + (((4 * at) ^ ((at >> 2) & 3) ^ swz_i(ai)) << 3) : -1;
                        ts[u] = at;
                        ai += DI;
                        at += DT;
                        sp += s1;
                        tp += t1;
                        if (DT && at >= PR) {
                            at -= PR;
                            ++ai;
                            sp += s2;
                            tp += t2;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < Sh::UA; ++u) {
                        if (clean) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) z[u][j].x = isfinite(z[u][j].x) ? z[u][j].x : 0.f;
                        }
                        float2 v[4];
                        if (q == 0) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) v[j] = cadd(z[u][j], z[u][j + 4]);
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j) v[j] = twiddle<-1>(csub(z[u][j], z[u][j + 4]), j, 8);
                        }
                        dft<4, -1>(v);
                        const float2* const tw = twr + 4 * q * PR + ts[u];
                        if (offs[u] >= 0) {
#pragma unroll
                            for (int k1 = 0; k1 < 4; ++k1) z_at(offs[u] ^ (k1 << 3)) = cmul(v[k1], tw[k1 * PR]);
                        }
                    }
                }
                __syncwarp();
                // ---- B: rows, radix PR
                for (int it = lane; it < rows * 4; it += 32) {
                    const int i = it >> 2, k1 = it & 3;
                    const int o = (rw + PC * i) * ZB + ((k1 ^ swz_i(i)) << 3);
                    float2 v[PR];
#pragma unroll
                    for (int t = 0; t < PR; ++t) v[t] = z_at((o ^ ((swz_c(4 * t) & 15) << 3)) + ((4 * t & ~15) << 3));
                    dft<PR, -1>(v);
#pragma unroll
                    for (int t = 0; t < PR; ++t) {
                        if (t >= PR / 2) v[t].y = -v[t].y;
                        z_at((o ^ ((swz_c(4 * t) & 15) << 3)) + ((4 * t & ~15) << 3)) = v[t];
                    }
                }
                __syncthreads();
                // ---- C: columns, radix 16
                const int Lc = s_it.Lw;
                // the next channel's rows on their way to L2 (a window's lines come from
                // HBM the first time; the row loads above wait for them)
                if (q == 1 && c + 1 < s_it.nch) {
                    constexpr int E = 128 / sizeof(T);  // elements per line
                    const int ns = (Lc + 2 * E - 2) / E, mt = s_it.m, nt = (mt + 2 * E - 2) / E;
                    const T* const Sn = s_it.S + (size_t)(c + 1) * s_it.splane;
                    const T* const Tn = s_it.T0 + (size_t)(c + 1) * s_it.tplane;
                    for (int i = tid; i < Lc * ns; i += NT) {
                        const int y = i / ns, x = min((i - y * ns) * E, Lc - 1);
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(Sn + (size_t)y * s_it.spitch + x));
                    }
                    for (int i = tid; i < mt * nt; i += NT) {
                        const int y = i / nt, x = min((i - y * nt) * E, mt - 1);
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(Tn + (size_t)y * s_it.tpitch + x));
                    }
                }
                for (int it = tid; it < Lh * PC; it += NT) {
                    const int t = it / Lh, col = it - t * Lh;
                    const int o = t * ZB + (swz_c(col) << 3);
                    float2 v[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        if (PC * j + PC - 1 < Sh::LMIN || t + PC * j < Lc) v[j] = z_at((o ^ (swz_i(j) << 3)) + PC * j * ZB);
                        else v[j] = make_float2(0.f, 0.f);
                    }
                    dft<16, -1>(v);
                    z_at(o) = v[0];
                    const float2* const tw = twc + t;
#pragma unroll
                    for (int k1 = 1; k1 < 16; ++k1) z_at((o ^ (swz_i(k1) << 3)) + PC * k1 * ZB) = cmul(v[k1], tw[k1 * PC]);
                }
                __syncthreads();
                // ---- D: columns, radix PC, in conjugate pairs; cross spectrum
#pragma unroll
                for (int r = 0; r < NI; ++r) {
                    const int it = tid + r * NT;
                    const int k1 = it / (Lh / 2), col = it - k1 * (Lh / 2);
                    const bool selfc = q == 0 && col == 0;
                    const int par = q ? Lh - 1 - col : (col ? Lh - col : Lh / 2);
                    const int oa = PC * k1 * ZB + ((swz_c(col) ^ swz_i(k1)) << 3);
                    const int ob = PC * k1 * ZB + ((swz_c(par) ^ swz_i(k1)) << 3);
                    float2 a[PC], b[PC];
#pragma unroll
                    for (int t = 0; t < PC; ++t) a[t] = z_at(oa + t * ZB);
#pragma unroll
                    for (int t = 0; t < PC; ++t) b[t] = z_at(ob + t * ZB);
                    dft<PC, -1>(a);
                    dft<PC, -1>(b);
                    if (selfc) {
#pragma unroll
                        for (int j = 0; j < PC; ++j) {
                            ex[k1 + 16 * j] = a[j];
                            ex[L + k1 + 16 * j] = b[j];
                        }
                    }
                    // (the sums of column 0's lanes are not used: add_self has its own)
                    float2 acc[PC];
                    tm_wait_st();
                    tm_load(tacc + q * Sh::tm_half + r * 2 * PC, acc);
                    tm_wait_ld();
#pragma unroll
                    for (int j = 0; j < PC; ++j) cross_add(acc[j], a[j], b[j]);
                    tm_store(tacc + q * Sh::tm_half + r * 2 * PC, acc);
                }
                __syncthreads();
                // (the next writes to ex are two barriers away)
                if (q == 0) add_self();
            }
        }
        __syncthreads();
        if (tid < 2 * L) ex[tid] = self;
        __syncthreads();
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
            // ---- inverse along the columns: PC-point over k2, twiddle ...
#pragma unroll
            for (int r = 0; r < NI; ++r) {
                const int it = tid + r * NT;
                const int k1 = it / (Lh / 2), col = it - k1 * (Lh / 2);
                float2 acc[PC];
                tm_wait_st();
                tm_load(tacc + q * Sh::tm_half + r * 2 * PC, acc);
                tm_wait_ld();
                if (q == 0 && col == 0) {
#pragma unroll
                    for (int j = 0; j < PC; ++j) acc[j] = ex[k1 + 16 * j];
                }
                dft<PC, 1>(acc);
                const int oa = PC * k1 * ZB + ((swz_c(col) ^ swz_i(k1)) << 3);
#pragma unroll
                for (int t = 0; t < PC; ++t) z_at(oa + t * ZB) = cmul_conj(acc[t], twc[k1 * PC + t]);
            }
            if (q == 0 && tid < 16) {  // column Lh / 2
                const int k1 = tid;
                float2 v[PC];
#pragma unroll
                for (int j = 0; j < PC; ++j) v[j] = ex[L + k1 + 16 * j];
                dft<PC, 1>(v);
#pragma unroll
                for (int t = 0; t < PC; ++t)
                    z_at((t + PC * k1) * ZB + ((swz_c(Lh / 2) ^ swz_i(k1)) << 3)) = cmul_conj(v[t], twc[k1 * PC + t]);
            }
            __syncthreads();
            // ... then 16-point over k1: rows t + PC j
            {
                const int cw = Lh / 2 + (q == 0 ? 1 : 0), P1 = s_it.P1;
                for (int it = tid; it < cw * PC; it += NT) {
                    const int t = it / cw, col = it - t * cw;
                    const int o = t * ZB + (swz_c(col) << 3);
                    float2 v[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = z_at((o ^ (swz_i(j) << 3)) + PC * j * ZB);
                    dft<16, 1>(v);
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (t + PC * j < P1) z_at((o ^ (swz_i(j) << 3)) + PC * j * ZB) = v[j];
                }
            }
            __syncthreads();
            // ---- inverse along the wanted rows (Hermitian extension), real part
            {
                const int P1 = s_it.P1;
                float* const out = s_it.out;
                const int orows = min(max((P1 - rw + PC - 1) / PC, 0), RI);
                const float scale = 0.25f / ((float)L * (float)L);
                bool bad = false;
                // every lane of the warp takes part in each round of 8 rows
                for (int i8 = 0; i8 < orows; i8 += 8) {
                    const int il = i8 + (lane >> 2), i = il, k1 = lane & 3, y = rw + PC * i;
                    const bool on = il < orows;
                    float2 v[PR];
                    if (on) {
#pragma unroll
                        for (int k2 = 0; k2 < PR; ++k2) {
                            const int kp = k1 + 4 * k2;
                            const bool up = kp >= Lh / 2 && !(q == 0 && kp == Lh / 2);
                            const int cc = up ? (q ? Lh - 1 - kp : Lh - kp) : kp;
                            v[k2] = z_at(y * ZB + ((swz_c(cc) ^ swz_i(i)) << 3));
                            if (up) v[k2].y = -v[k2].y;
                        }
                        dft<PR, 1>(v);
                    }
                    __syncwarp();
                    if (on) {
                        const int o = y * ZB + ((k1 ^ swz_i(i)) << 3);
#pragma unroll
                        for (int t = 0; t < PR; ++t)
                            z_at((o ^ ((swz_c(4 * t) & 15) << 3)) + ((4 * t & ~15) << 3)) =
                                cmul_conj(v[t], twr[(4 * q + k1) * PR + t]);
                    }
                    __syncwarp();
                    for (int it = lane; it < 8 * PR; it += 32) {
                        const int i2 = i8 + it / PR, t = it % PR;
                        if (i2 >= orows) break;
                        const int yy = rw + PC * i2;
                        const int o = yy * ZB + (((4 * t) ^ ((t >> 2) & 3) ^ swz_i(i2)) << 3);
                        float2 u[4];
#pragma unroll
                        for (int a = 0; a < 4; ++a) u[a] = z_at(o ^ (a << 3));
                        dft<4, 1>(u);
                        float* const orow = out + (size_t)yy * P1;
#pragma unroll
                        for (int x1 = 0; x1 < 4; ++x1) {
                            const float2 w = q ? twiddle<1>(u[x1], x1, 8) : u[x1];
                            const float val = w.x * scale;
                            bad = bad || !isfinite(val);
                            const int x = t + PR * x1;
                            if (x < P1) orow[x] = q ? orow[x] + val : val;
                            if (x + Lh < P1) orow[x + Lh] = q ? orow[x + Lh] - val : val;
                        }
                    }
                    __syncwarp();
                }
                // a non-finite value of the window may not reach the offsets whose windows
                // do not hold it (the tensor-core forms keep it apart too, and which form a
                // window gets is a matter of measured time): once more, with zeros in its
                // place
                if (__syncthreads_or(bad && !clean)) again = true;
            }
            if (again) break;
        }
        clean = again;
    }
    tm_wait_st();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Sh::tm_cols) : "memory");
}

}  // namespace

int corr_fft2_side(int m, int R) {
    const int lw = m + 2 * R;
    if (lw <= 64 || (lw > 96 && lw <= 128) || lw > 224) return 0;
    return (lw + 31) / 32 * 32;
}

cudaError_t launch_corr_fft2(const MatchJob& one, const ItemSet& is, int L, bool bf16, cudaStream_t st) {
    const int n = is.items ? is.n : one.n;
    if (n <= 0) return cudaSuccess;
    if (!is.items && (bf16 ? (one.rpl == nullptr || one.spl == nullptr || one.z != 12)
                           : (one.rf32 == nullptr || one.sf32 == nullptr)))
        return cudaErrorNotSupported;
    const int lw = one.m + 2 * one.R;
    if (!is.items && (lw > L || lw <= L - 32)) return cudaErrorNotSupported;
    const int sms = device_sms();
    auto run = [&](auto kern, auto shape) -> cudaError_t {
        using Sh = decltype(shape);
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem);
        if (e != cudaSuccess) return e;
        const int ctas = sms * Sh::MINB;
        kern<<<n < ctas ? n : ctas, Sh::NT, Sh::smem, st>>>(one, is.jobs, is.items, n, is.queue);
        return cudaGetLastError();
    };
    switch (L) {
#define SFOC_FFT_SIDE(LV)                                                              \
    case LV:                                                                           \
        return bf16 ? run(k_corr_fft2<LV, __nv_bfloat16>, FftShape<LV>())              \
                    : run(k_corr_fft2<LV, float>, FftShape<LV>());
        SFOC_FFT_SIDE(96)
        SFOC_FFT_SIDE(160)
        SFOC_FFT_SIDE(192)
        SFOC_FFT_SIDE(224)
#undef SFOC_FFT_SIDE
        default: return cudaErrorNotSupported;
    }
}

}  // namespace sfoc

// AX operator to FP64 accuracy on the integer and FP32 pipes: the line-pass kernel of nx >= 5.
//
// The operator is Section II-B's, Listing 1 of arXiv 2011.04981: w = D^T (G (D u)) per element.  Every contraction
// along a line of nx points is done in block fixed point:
//   - the element's values are scaled by a power of two to below 2^28 and split into an integer digit (the
//     nearest integer of the float pair's high part) and the float remainder, at most 2^-24 of the largest value;
//   - D is scaled and split the same way (26 bits of its row's absolute sum in phase 1, 27 of the whole matrix in phase 2);
//   - digit x digit products are summed exactly in 64-bit integers (IMAD.WIDE: 64 a clock and SM, measured), the
//     two cross products with the remainders in floats (packed FFMA2).
// A term costs three multiply-adds; the float-float form with tracked residuals (k_ax_ff) takes nine.
//   - D of a symmetric rule satisfies D[n-1-i][n-1-l] = -D[i][l].  With the sums and differences of mirrored points
//     (exact in integers) every product serves two outputs, which halves the multiply-adds and the loads of D.  The
//     kernel checks the symmetry of the D it is given, exactly, and otherwise computes every row for itself.
// The geometric product at a point takes the derivatives as float pairs and sums each row at an offset
// (fx_dot3).  The phase-2 sums of the three directions share one scale, are added as integers and joined to a double at the
// end.  Errors against 64 bits (2-norm, random u, deformed boxes): 1.6e-14 at nx = 5, 2.0e-14 at 10, 2.4e-14 at 16 (the
// float-float kernels before it 6.9e-14, 1.7e-13, 2.8e-13).  22-bit digits by the addition of 1.5 2^23 instead of the
// conversion instruction gave 8e-14 for 2 % less time; not taken.
//
// Mapping: a thread owns two (or one, fx_lpt) of the element's 3 nx^2 lines, holds their points in registers and writes all
// their outputs, so a point is read once per direction and phase and D is read as broadcasts.  The point-wise stages
// (input, G, result) run over the same threads, point t, t + TPE, ...  CTAs are persistent: the tables of D are
// built once, the next element's input is copied to shared memory (cp.async, in the place of the split
// form) under the current one's second half, and the element's G is fetched into L2 while phase 1 runs.
//
// What bounds it (nx = 10, 32768 elements, ncu): no unit is saturated; issue 52 %, shared-memory data path 61 %, FMA
// pipes 36 %; the 4.8 warps a scheduler wait on fixed latencies, global loads, shared loads and barriers in about equal
// parts.  0.61 ms = 53 GDOF/s = 0.50 of the measured HBM copy rate at 64 B/point (float-float item kernel before: 0.96
// ms); with the solve's direction update 0.80 ms = 0.62 of it at 104 B/point (1.04 ms before).
#pragma once

#include <type_traits>

#include "nek_ff.cuh"
#include "nek_internal.h"
#include "nek_lines.cuh"
#include "nek_pdl.cuh"
#include "nek_reduce.cuh"

namespace nek {

namespace {

// Lines per thread (of the 3 nx^2 lines of a phase), resident warps per SM that the register budget is set for, and points
// whose geometric factors are in flight together.  Two lines a thread halve the loads of the matrix tables; at nx = 11,
// 12 and 14 one line with more warps measured faster (nx = 12: 0.71 against 0.74 ms plain, 0.92 against 0.98 with the
// direction update, a 30-million-point launch).  Warps (us, plain, 8 million points): nx = 6 145 with 28, 148 with 20; 8 139
// with 24, 149 with 20, 151 with 28; 11 193 with 36, 191 with 28, 242 with 20; 12 183 with 28, 231 with 24; at the others 20,
// where 16 is slower or the same (nx = 5 172 and 193, 7 169 and 182) and 28 is slower (9 162 and 191, 10 156 and 201, which
// spills) or makes no difference (from 13 on: shared memory).  Points of G together, 2 or 3 (with energies): nx = 8 153 and
// 149, 10 no difference, 6, 9 and 12 to 14 two to 6 % slower with three (9: 170 and 176).
constexpr int fx_lpt(int nx) { return nx == 11 || nx == 12 || nx == 14 ? 1 : 2; }
constexpr int fx_warps(int nx) { return nx == 6 || nx == 12 ? 28 : nx == 8 ? 24 : nx == 11 ? 36 : 20; }
constexpr int fx_ahead(int nx) { return nx == 8 || nx == 10 ? 3 : 2; }
// Bits of the digits: values (sum and difference of two: one more), D in phase 1 (whose rows' absolute sums stay below
// 2^kBits1, so a row's result stays below 2^54: 24 bits and 30 more) and in phase 2, and the power of two that
// keeps phase 2's float cross sums (at most 16 (2^27 + 17 2^27)) within a 32-bit integer.
constexpr int kBitsU = 28, kBits1 = 26, kBits2 = 27, kCrossShift = 6;
// Threads per element and per CTA of epb elements.
constexpr int fx_tpe(int nx) { return (3 * nx * nx + fx_lpt(nx) - 1) / fx_lpt(nx); }
constexpr int fx_threads(int nx, int epb) { return (fx_tpe(nx) * epb + 31) / 32 * 32; }

template <int NX>
struct FxTab {
    static constexpr int HE = (NX + 1) / 2, NI = (2 * HE + 3) / 4 * 4;
    float4 f[NX * HE];  // row i, entry l: remainders (even, odd) and values (even, odd) of the folded matrix
    int d[NX * NI];     // row i: the integer digits (even, odd) of entry l at 2 l
};

template <int NX, int EPB>
struct FxSmem {
    static constexpr int NP = FxGrid<NX>::SIZE;
    float2 U[EPB * NP];
    float2 A[3][EPB * NP];  // gradient / products (float pairs), then the line sums of phase 2 (64-bit integers)
    FxTab<NX> t1, t2;
    float rs[NX];           // phase 1: value of one unit of row i's sums
    unsigned mx[2][2 * (EPB + 1)];  // per element: bits of max |u|, of max |wr|, |ws|, |wt|; two buffers
    int dexp[NX];      // exponents above row i's absolute sum
    unsigned dmax;     // high word of the largest entry's magnitude
    double esum[fx_threads(NX, EPB)];
};

constexpr unsigned kInfBits = 0x7F800000u;

// Pairs of floats kept as one 64-bit register pair, so that no packing moves are issued at their uses.
typedef unsigned long long f32pair;
__device__ __forceinline__ f32pair pk(float a, float b)
{
    f32pair r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpk(f32pair p, float& a, float& b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
}
__device__ __forceinline__ f32pair ffma2(f32pair a, f32pair b, f32pair c)
{
    f32pair r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32pair fmul2(f32pair a, f32pair b)
{
    f32pair r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// 2^e as a float, e clamped to the normal range.
__device__ __forceinline__ float pow2f(int e)
{
    e = e < -126 ? -126 : e > 127 ? 127 : e;
    return __int_as_float((e + 127) << 23);
}

// split_double with infinities, NaNs and values beyond the float range made infinite: h the top 24 significant
// bits, l the next 23, both with the sign of x.
__device__ __forceinline__ float2 fx_split(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned a = hi & 0x7FFFFFFFu, sgn = hi & 0x80000000u;
    unsigned h = (__funnelshift_l(lo, hi, 3) - (896u << 23)) & 0x7FFFFFFFu;
    h = a >= (1151u << 20) ? kInfBits : h;
    const float r = __fsub_rn(__uint_as_float(0x4B000000u | ((lo >> 6) & 0x7FFFFFu)), 8388608.0f);
    // r times 2^(e - 1069) with x's sign; below 2^-80 no low part, below 2^-126 nothing
    const unsigned s = ((a & 0x7FF00000u) << 3) - (942u << 23);
    const float l = a >= (943u << 20) ? __fmul_rn(r, __uint_as_float(s | sgn)) : 0.f;
    return make_float2(__uint_as_float(a >= (897u << 20) ? h | sgn : 0u), l);
}

// The same for any exponent (overflow to infinity, underflow to zero).
__device__ __forceinline__ double fx_ldexp_any(long long z, int x)
{
    const double v = fx_ldexp(z, 0);
    const unsigned hi = (unsigned)__double2hiint(v);
    const int e = (int)((hi >> 20) & 0x7FFu) + x;
    if (z == 0 || e <= 0) return 0.0;
    if (e >= 0x7FF) return __hiloint2double((int)((hi & 0x80000000u) | 0x7FF00000u), 0);
    return __hiloint2double((int)(hi + ((unsigned)x << 20)), __double2loint(v));
}

// The folded matrix of one phase.  M = D (phase 1) or D^T (phase 2).  Row i, entry l < ceil(n/2): the even part
// multiplies u_l + u_{n-1-l} (the middle point alone where n is odd), the odd part u_l - u_{n-1-l}.  Values are
// scaled by 2^(bits - E) with 2^E above the row's absolute sum (PER_ROW) or the matrix's largest entry, and split into
// the nearest integer and the float remainder; the float forms are multiplied by s: the value of one unit of the row's
// sums (PER_ROW) or 2^-kCrossShift.  Entry q = i ceil(n/2) + l of the table, e its E.
template <int NX, bool PER_ROW>
__device__ __forceinline__ void fx_entry(const double* Ds, int q, int e, float s, FxTab<NX>& t)
{
    constexpr int HE = FxTab<NX>::HE, kBits = PER_ROW ? kBits1 : kBits2;
    const int i = q / HE, l = q - i * HE, m = NX - 1 - l;
    const double a = PER_ROW ? Ds[i * NX + l] : Ds[l * NX + i];
    const double b = PER_ROW ? Ds[i * NX + m] : Ds[m * NX + i];
    const double sc = __hiloint2double((1023 + kBits - e) << 20, 0);
    const double ve = (l == m ? a : 0.5 * (a + b)) * sc, vo = (l == m ? 0.0 : 0.5 * (a - b)) * sc;
    const int de = __double2int_rn(ve), dd = __double2int_rn(vo);
    t.f[q] = make_float4((float)(ve - (double)de) * s, (float)(vo - (double)dd) * s, (float)de * s, (float)dd * s);
    t.d[i * FxTab<NX>::NI + 2 * l] = de;
    t.d[i * FxTab<NX>::NI + 2 * l + 1] = dd;
}

// Both tables, an entry a thread.  An FP64 instruction takes a warp 64 clocks: the tables one after the other, and the
// largest entry by a chain of nx^2 maxima in one thread, made every call 5 us longer at nx = 10 and 14 at nx = 16 (64
// elements: nx = 10 15.0 -> 9.4 us, 8 10.8 -> 6.7, 16 32.6 -> 18.4).
template <int NX>
__device__ __forceinline__ void fx_build(const double* Ds, const int* dexp, int ED, FxTab<NX>& t1, FxTab<NX>& t2, int tid,
                                         int nt)
{
    constexpr int N = NX * FxTab<NX>::HE;
    for (int q = tid; q < 2 * N; q += nt) {
        if (q < N) {
            const int e = dexp[q / FxTab<NX>::HE];
            fx_entry<NX, true>(Ds, q, e, pow2f(e - kBitsU - kBits1), t1);
        } else {
            fx_entry<NX, false>(Ds, q - N, ED, 1.f / (1 << kCrossShift), t2);
        }
    }
}

// One line pass over LPT lines of NX points: src[q] and dst[q] hold NX values at stride st[q].
//   phase 1: dst = float pair of sum_l D[i][l] u_l (units of 2^E, the element's scale)
//   phase 2: dst = the sum as a 64-bit integer
template <int NX, int PHASE, int LPT>
__device__ __forceinline__ void fx_lines(const float2* const (&src)[LPT], float2* const (&dst)[LPT],
                                         const int (&st)[LPT], const float (&sg)[LPT], float scale, const FxTab<NX>& tab,
                                         const float* __restrict__ rs, bool sym)
{
    constexpr int HE = FxTab<NX>::HE, HO = NX / 2, NI = FxTab<NX>::NI;
    int dg[LPT][2 * HE];                       // digits: sum and difference of points l and n-1-l
    f32pair df[LPT][HE], lf[LPT][HE];           // (sum, difference) of the digits as floats, and of the remainders
#pragma unroll
    for (int q = 0; q < LPT; q++) {
        const float sc = sg[q] * scale;
        // digit, digit as a float (its nearest 24 bits where it has more: then the value itself), remainder
        auto conv = [&](float2 a, int& d, float& h, float& l) {
            const float hs = __fmul_rn(a.x, sc);
            d = __float2int_rn(hs);
            h = __int2float_rn(d);
            l = __fmaf_rn(a.y, sc, __fsub_rn(hs, h));
        };
#pragma unroll
        for (int l = 0; l < HE; l++) {
            const int m = NX - 1 - l;
            int d;
            float h, r;
            conv(src[q][l * st[q]], d, h, r);
            if (l == m) {
                dg[q][2 * l] = d;
                dg[q][2 * l + 1] = 0;
                df[q][l] = pk(h, 0.f);
                lf[q][l] = pk(r, 0.f);
            } else {
                int d2;
                float h2, r2;
                conv(src[q][m * st[q]], d2, h2, r2);
                dg[q][2 * l] = d + d2;
                dg[q][2 * l + 1] = d - d2;
                df[q][l] = pk(__fadd_rn(h, h2), __fsub_rn(h, h2));
                lf[q][l] = pk(__fadd_rn(r, r2), __fsub_rn(r, r2));
            }
        }
    }
    auto put = [&](int q, int i, long long y, float cr) {
        if constexpr (PHASE == 1) {
            const float s = rs[i], t = (float)(int)(y >> 30), K = s * 1073741824.f;
            const float l = __fmaf_rn((float)((unsigned)y & 0x3FFFFFFFu), s, cr);
            dst[q][i * st[q]] = make_float2(t * K, l);
        } else {
            *reinterpret_cast<long long*>(dst[q] + i * st[q]) = madw(__float2int_rn(cr), 1 << kCrossShift, y);
        }
    };
    auto row = [&](int i, long long (&a)[LPT], long long (&b)[LPT], f32pair (&c)[LPT]) {
        const ulonglong2* f = reinterpret_cast<const ulonglong2*>(tab.f + i * HE);
        const int4* dq = reinterpret_cast<const int4*>(tab.d + i * NI);
        int4 v4;
#pragma unroll
        for (int l = 0; l < HE; l++) {
            if ((l & 1) == 0) v4 = dq[l >> 1];
            const int de = (l & 1) ? v4.z : v4.x, dd = (l & 1) ? v4.w : v4.y;
            const ulonglong2 v = f[l];
#pragma unroll
            for (int q = 0; q < LPT; q++) {
                a[q] = l == 0 ? (long long)dg[q][0] * de : madw(dg[q][2 * l], de, a[q]);
                if (l == 0)
                    b[q] = (long long)dg[q][1] * dd;
                else if (2 * l != NX - 1)
                    b[q] = madw(dg[q][2 * l + 1], dd, b[q]);
                c[q] = l == 0 ? fmul2(df[q][0], v.x) : ffma2(df[q][l], v.x, c[q]);
                c[q] = ffma2(lf[q][l], v.y, c[q]);
            }
        }
    };
    if (sym) {
#pragma unroll 1
        for (int i = 0; i < HE; i++) {
            long long a[LPT], b[LPT];
            f32pair c[LPT];
            row(i, a, b, c);
#pragma unroll
            for (int q = 0; q < LPT; q++) {
                float ce, co;
                unpk(c[q], ce, co);
                put(q, i, a[q] + b[q], __fadd_rn(ce, co));
                if (HE == HO || i < HO) put(q, NX - 1 - i, b[q] - a[q], __fsub_rn(co, ce));
            }
        }
    } else {
#pragma unroll 1
        for (int i = 0; i < NX; i++) {
            long long a[LPT], b[LPT];
            f32pair c[LPT];
            row(i, a, b, c);
#pragma unroll
            for (int q = 0; q < LPT; q++) {
                float ce, co;
                unpk(c[q], ce, co);
                put(q, i, a[q] + b[q], __fadd_rn(ce, co));
            }
        }
    }
}

// (ah + al)(x.x + x.y) + (bh + bl)(y.x + y.y) + (ch + cl)(z.x + z.y) as an unevaluated pair.  The running sum S
// starts at an offset whose binade holds every partial sum (1.5 * 2^m, 2^m above the sum of the terms'
// magnitudes), so S - t is exact and each product's remainder is one fused multiply-add.
__device__ __forceinline__ void fx_dot3(float ah, float al, float2 x, float bh, float bl, float2 y, float ch, float cl,
                                        float2 z, float2& w)
{
    const float B = __fmaf_rn(fabsf(ch), fabsf(z.x), __fmaf_rn(fabsf(bh), fabsf(y.x), __fmul_rn(fabsf(ah), fabsf(x.x))));
    const float s0 = offset_for(B);
    const float t1 = __fmaf_rn(ah, x.x, s0);
    const float r1 = __fmaf_rn(ah, x.x, __fsub_rn(s0, t1));
    const float t2 = __fmaf_rn(bh, y.x, t1);
    const float r2 = __fmaf_rn(bh, y.x, __fsub_rn(t1, t2));
    const float t3 = __fmaf_rn(ch, z.x, t2);
    const float r3 = __fmaf_rn(ch, z.x, __fsub_rn(t2, t3));
    const float c1 = __fmaf_rn(al, x.x, __fmaf_rn(ah, x.y, r1));
    const float c2 = __fmaf_rn(bl, y.x, __fmaf_rn(bh, y.y, r2));
    const float c3 = __fmaf_rn(cl, z.x, __fmaf_rn(ch, z.y, r3));
    const float h = __fsub_rn(t3, s0), l = __fadd_rn(__fadd_rn(c1, c2), c3), n = __fadd_rn(h, l);
    w = make_float2(n, __fsub_rn(l, __fsub_rn(n, h)));  // |w.y| <= 2^-24 |w.x| also where the terms cancel
}

// slot[key] = max(slot[key], v) over the block; every thread takes part.
template <int EPB>
__device__ __forceinline__ void fx_max(int key, unsigned v, unsigned* slot)
{
    if constexpr (EPB == 1) {
        const unsigned m = __reduce_max_sync(0xffffffffu, v);  // idle lanes of the last warp bring 0
        if ((threadIdx.x & 31) == 0) atomicMax(slot, m);
    } else {
        const unsigned same = __match_any_sync(0xffffffffu, key);
        const unsigned m = __reduce_max_sync(same, v);
        if ((threadIdx.x & 31) == __ffs(same) - 1) atomicMax(slot + key, m);
    }
}

template <int NX, int EPB>
constexpr int fx_min_blocks()
{
    const int by_smem = (int)((227 * 1024) / (sizeof(FxSmem<NX, EPB>) + 1024));
    const int by_warps = fx_warps(NX) / (fx_threads(NX, EPB) / 32);
    const int b = by_smem < by_warps ? by_smem : by_warps;
    return b < 1 ? 1 : b;
}

template <int NX, int EPB, int MODE>
__global__ void __launch_bounds__(fx_threads(NX, EPB), (fx_min_blocks<NX, EPB>()))
    k_ax_fx(int64_t nelt, const double* __restrict__ D, const float4* __restrict__ Gff,
            const double* __restrict__ u, double* __restrict__ w, const int32_t* __restrict__ l2g,
            const int32_t* __restrict__ eprob, const uint8_t* __restrict__ pdone, double* __restrict__ edot,
            DirUpdate dir)
{
    using Grid = FxGrid<NX>;
    constexpr int NP = Grid::SIZE, N2 = NX * NX, N3 = NX * NX * NX;
    constexpr int TPE = fx_tpe(NX), NT = fx_threads(NX, EPB), kAhead = fx_ahead(NX);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FxSmem<NX, EPB>& S = *reinterpret_cast<FxSmem<NX, EPB>*>(smem_raw);
    const int tid = threadIdx.x;

    // ---- the matrix tables, once per CTA
    bool sym, dbad;
    int ED;
    {
        double* Ds = reinterpret_cast<double*>(S.A);
        for (int q = tid; q < N2; q += NT) Ds[q] = D[q];
        if (tid < 2 * (EPB + 1)) S.mx[0][tid] = S.mx[1][tid] = 0u;
        if (tid == 0) S.dmax = 0u;
        __syncthreads();
        bool asym = false;
        unsigned hm = 0u;
        for (int q = tid; q < N2; q += NT) {
            asym = asym || Ds[q] != -Ds[N2 - 1 - q];
            hm = max(hm, (unsigned)__double2hiint(Ds[q]) & 0x7FFFFFFFu);
        }
        hm = __reduce_max_sync(0xffffffffu, hm);
        if ((tid & 31) == 0 && hm) atomicMax(&S.dmax, hm);
        if (tid < NX) {
            double m = 0.0;
            for (int l = 0; l < NX; l++) m += fabs(Ds[tid * NX + l]);
            const int e = max((__double2hiint(m) >> 20) - 1022, -100);
            S.dexp[tid] = e;
            S.rs[tid] = pow2f(e - kBitsU - kBits1);
        }
        sym = !__syncthreads_or(asym);
        ED = max((int)(S.dmax >> 20) - 1022, -100);
        dbad = ED >= 128;  // beyond the float range, infinite, NaN
        for (int l = 0; l < NX; l++) dbad = dbad || S.dexp[l] >= 132;
        fx_build<NX>(Ds, S.dexp, ED, S.t1, S.t2, tid, NT);
        __syncthreads();
    }

    const int el = tid / TPE, t = tid - el * TPE;
    // this thread's lines (line L: direction L / N2, line L % N2 of it), all of element el; a thread whose last
    // line would be past the end repeats its first
    constexpr int LPT = fx_lpt(NX);
    const float2* src1[LPT];
    float2* dstA[LPT];
    const float2* src2[LPT];
    int str[LPT];
    float sgn[LPT];
#pragma unroll
    for (int q = 0; q < LPT; q++) {
        const int L = t + q * TPE < 3 * N2 ? t + q * TPE : t;
        const int d = L / N2, c = L - d * N2, b = c / NX, a = c - b * NX;
        int base = (el < EPB ? el : 0) * NP +
                   (d == 0 ? a * Grid::ROW + b * Grid::PLANE : a + b * (d == 1 ? Grid::PLANE : Grid::ROW));
        str[q] = d == 0 ? 1 : d == 1 ? Grid::ROW : Grid::PLANE;
        sgn[q] = 1.f;
        if (Grid::REV != 0 && d == 0 && sym && (t / (Grid::REV ? Grid::REV : 1)) & 1) {
            base += NX - 1;
            str[q] = -1;
            sgn[q] = -1.f;
        }
        src1[q] = S.U + base;
        dstA[q] = S.A[d] + base;
        src2[q] = dstA[q];
    }
    int buf = 0;
    int64_t prev = -1;  // first element of the group whose energies are still to be summed
    // The element sums of the threads' energies (doubles in esum), by the last warps.  FP64 additions cost a
    // 64-cycle pass of the scheduler's FP64 pipe each, and the other warps wait for the result at the next barrier; so
    // the values are brought to the largest one's exponent as 64-bit integers (rounded to 2^-53 of it) and summed
    // exactly, in any order.
    auto flush_energies = [&]() {
        if constexpr (mode_energies(MODE)) {
            constexpr int NV = (TPE + 31) / 32;
            const int warp = tid >> 5, lane = tid & 31;
            if (prev >= 0) {
                for (int e = NT / 32 - 1 - warp; e < EPB; e += NT / 32) {
                    if (prev + e >= nelt) continue;
                    double v[NV];
                    unsigned mx = 0u;
#pragma unroll
                    for (int k = 0; k < NV; k++) {
                        v[k] = lane + 32 * k < TPE ? S.esum[e * TPE + lane + 32 * k] : 0.0;
                        mx = max(mx, (unsigned)__double2hiint(v[k]) & 0x7FF00000u);
                    }
                    const int em = (int)(__reduce_max_sync(0xffffffffu, mx) >> 20);
                    long long sum = 0;
#pragma unroll
                    for (int k = 0; k < NV; k++) {
                        const unsigned hi = (unsigned)__double2hiint(v[k]);
                        const int ex = (int)((hi >> 20) & 0x7FFu);
                        const unsigned long long mant =
                            ((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32) | (unsigned)__double2loint(v[k]);
                        const int sh = em - ex;
                        const long long f = ex == 0 || sh > 53 ? 0 : (long long)(((mant << 1 >> sh) + 1) >> 1);
                        sum += (int)hi < 0 ? -f : f;
                    }
                    // warp sum in three pieces that cannot overflow 32 bits
                    const unsigned p0 = __reduce_add_sync(0xffffffffu, (unsigned)(sum & 0x3FFFFFF));
                    const unsigned p1 = __reduce_add_sync(0xffffffffu, (unsigned)((sum >> 26) & 0x3FFFFFF));
                    const int p2 = __reduce_add_sync(0xffffffffu, (int)(sum >> 52));
                    const long long tot = ((long long)p2 << 52) + ((long long)p1 << 26) + (long long)p0;
                    if (lane == 0)
                        edot[prev + e] = em == 0x7FF ? __longlong_as_double(0x7FF8000000000000LL)
                                                     : em == 0 ? 0.0 : fx_ldexp_any(tot, em - 1023 - 52);
                }
            }
        }
    };
    // points of the element that this thread loads, multiplies with G and writes: t, t + TPE, ...
    constexpr int B = (N3 + TPE - 1) / TPE;
    constexpr bool DIR = MODE == kModeDirDot;
    bool dx = false, dp = false;
    double da = 0.0, db = 0.0;
    if constexpr (DIR) {
        pdl_wait(dir.sc);  // only the matrix has been read so far
        dx = dir.sc->xpend != 0;
        dp = !(dir.sc->done || dir.sc->status != NEK_OK);
        da = dir.sc->alpha;
        db = dir.sc->beta;
    }
    float2* Ue = S.U + (el < EPB ? el : 0) * NP;
    float2 *Ut = Ue + Grid::at(t), *At[3];  // this thread's first point
#pragma unroll
    for (int d = 0; d < 3; d++) At[d] = S.A[d] + (el < EPB ? el : 0) * NP + Grid::at(t);
    // offset of its b-th point from them (a constant on the dense grids)
    auto off = [&](int b) {
        if constexpr (Grid::ROW == NX && Grid::PAD == 0)
            return b * TPE;
        else
            return Grid::at(t + b * TPE) - Grid::at(t);
    };
    auto has = [&](int b) { return b < B - 1 || t + b * TPE < N3; };
    // Starts copying the group's input (raw doubles, each thread its own points) to shared memory: u or p to the
    // places of their split form; the direction update's other inputs are fetched into L2.
    auto fetch = [&](int64_t g0) {
        if (el < EPB && g0 + el < nelt) {
            const int64_t gf = (g0 + el) * (int64_t)N3 + t;
            const double* src = DIR ? dir.p + gf : u + gf;
            const int32_t* idx = mode_gathers(MODE) ? l2g + gf : nullptr;
#pragma unroll
            for (int b = 0; b < B; b++)
                if (has(b)) cp_async8(Ut + off(b), mode_gathers(MODE) ? u + __ldg(idx + b * TPE) : src + b * TPE);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if constexpr (DIR) {
            if (tid == 0) {
                const int64_t n = (nelt - g0 < EPB ? nelt - g0 : EPB) * (int64_t)N3;
                l2_prefetch(dir.x + g0 * N3, n);
                l2_prefetch(dir.minv + g0 * N3, n);
                l2_prefetch(dir.r + g0 * N3, n);
            }
        }
    };
    // DIR: x, minv and r of the thread's b-th point (g: its first point of the next group) into its own, then free,
    // places of A
    auto fetch_dir = [&](int64_t g, int b) {
        if constexpr (DIR) {
            cp_async8(At[0] + off(b), dir.x + g + b * TPE);
            cp_async8(At[1] + off(b), dir.minv + g + b * TPE);
            cp_async8(At[2] + off(b), dir.r + g + b * TPE);
        }
    };
    // the next group of elements from e0 on that has work (e0 >= nelt: none left)
    const int64_t step = (int64_t)gridDim.x * EPB;
    auto group_from = [&](int64_t e0) {
        while (e0 < nelt &&
               cta_skipped<MODE>(eprob, pdone, e0, static_cast<int>(nelt - e0 < EPB ? nelt - e0 : EPB)))
            e0 += step;
        return e0;
    };
    int64_t e0 = group_from((int64_t)blockIdx.x * EPB);
    if (e0 < nelt) {
        fetch(e0);
        if constexpr (DIR) {
            if (el < EPB && e0 + el < nelt) {
                for (int b = 0; b < B; b++)
                    if (has(b)) fetch_dir((e0 + el) * (int64_t)N3 + t, b);
            }
        }
    }
    while (e0 < nelt) {
        const int ne = static_cast<int>(nelt - e0 < EPB ? nelt - e0 : EPB);
        const bool active = el < ne;
        const int64_t ef = (e0 + el) * (int64_t)N3;  // the element's first point
        const int64_t enext = group_from(e0 + step);
        if (tid == 0) {  // the group's geometric factors into L2, needed after phase 1
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(Gff + e0 * N3 * 3),
                         "r"((unsigned)(ne * N3 * 48))
                         : "memory");
        }
        // ---- input: the direction update, split into float pairs (in place), element maximum
        {
            unsigned m = 0u;
            asm volatile("cp.async.wait_all;" ::: "memory");
            if (active) {
                double *xt = nullptr, *pt = nullptr;
                if constexpr (DIR) {
                    xt = dir.x + ef + t;
                    pt = dir.p + ef + t;
                }
#pragma unroll
                for (int b = 0; b < B; b++) {
                    if (has(b)) {
                        double v = *reinterpret_cast<const double*>(Ut + off(b));
                        if constexpr (DIR) {
                            if (dx) xt[b * TPE] = fma(da, v, *reinterpret_cast<const double*>(At[0] + off(b)));
                            if (dp) {
                                v = fma(db, v, *reinterpret_cast<const double*>(At[1] + off(b)) *
                                                   *reinterpret_cast<const double*>(At[2] + off(b)));
                                pt[b * TPE] = v;
                            }
                        }
                        const float2 s = fx_split(v);
                        Ut[off(b)] = s;
                        m = max(m, __float_as_uint(s.x) & 0x7FFFFFFFu);
                    }
                }
            }
            fx_max<EPB>(el < EPB ? el : EPB, m, S.mx[buf]);
        }
        __syncthreads();
        flush_energies();
        const unsigned mu = S.mx[buf][el < EPB ? el : EPB];
        const int eu = max((int)(mu >> 23), 28) - 126;  // 2^eu above the element's |u|
        // ---- phase 1: derivatives along the lines
        if (active) fx_lines<NX, 1, LPT>(src1, dstA, str, sgn, pow2f(kBitsU - eu), S.t1, S.rs, sym);
        __syncthreads();
        if (enext < nelt) fetch(enext);  // U is free: every line has been read
        // ---- geometric factors
        {
            unsigned m = 0u;
            if (active) {
                const float4* gp = Gff + (ef + t) * 3;
                int p = t;
                auto point = [&](int d, int a) {  // d points after the loop's p, a its place from the first point's
                    const float4 g0 = __ldg(gp + 3 * d), g1 = __ldg(gp + 3 * d + 1), g2 = __ldg(gp + 3 * d + 2);
                    const float2 r = At[0][a], s = At[1][a], q = At[2][a];
                    float2 w0, w1, w2;
                    fx_dot3(g0.x, g0.y, r, g0.z, g0.w, s, g1.x, g1.y, q, w0);
                    fx_dot3(g0.z, g0.w, r, g1.z, g1.w, s, g2.x, g2.y, q, w1);
                    fx_dot3(g1.x, g1.y, r, g2.x, g2.y, s, g2.z, g2.w, q, w2);
                    At[0][a] = w0;
                    At[1][a] = w1;
                    At[2][a] = w2;
                    m = max(max(m, __float_as_uint(fabsf(w0.x))),
                            max(__float_as_uint(fabsf(w1.x)), __float_as_uint(fabsf(w2.x))));
                };
#pragma unroll kAhead
                for (; p < N3; p += TPE, gp += 3 * TPE) point(0, Grid::at(p) - Grid::at(t));
            }
            fx_max<EPB>(el < EPB ? el : EPB, m, S.mx[buf] + EPB + 1);
        }
        __syncthreads();
        const unsigned mw = S.mx[buf][(el < EPB ? el : EPB) + EPB + 1];
        const int ew = max((int)(mw >> 23), 28) - 126;
        // ---- phase 2: transposed contraction along the lines, in place
        if (active) fx_lines<NX, 2, LPT>(src2, dstA, str, sgn, pow2f(kBitsU - ew), S.t2, S.rs, sym);
        if (tid < 2 * (EPB + 1)) S.mx[buf ^ 1][tid] = 0u;
        __syncthreads();
        // ---- sum of the three directions, joined to FP64
        double energy = 0.0;
        if (active) {
            double ue[mode_energies(MODE) ? B : 1];
            if constexpr (mode_energies(MODE)) {
#pragma unroll
                for (int b = 0; b < B; b++)
                    ue[b] = reread_input<MODE>(ef + t, has(b) ? b * TPE : 0, u, l2g, dir);
            }
            // (double)z 2^X for a 64-bit integer z: (2^84 + 2^63 + its high word) and (2^52 + its low word), both exact,
            // subtracted and summed, with X added to every exponent
            const int x = eu + ew + ED - kBitsU - kBits2, X = x << 20;
            const bool bad = dbad || mu >= kInfBits || mw >= kInfBits;
            const double C = bad ? __longlong_as_double(0x7FF8000000000000LL)
                                 : __hiloint2double(0x45300000 + X, 0x80100000);
            double* we = w + ef + t;
            const bool more = enext + el < nelt;
            const int64_t gn = (enext + el) * (int64_t)N3 + t;
#pragma unroll
            for (int b = 0; b < B; b++) {
                if (has(b)) {
                    auto Z = [&](int d) { return *reinterpret_cast<const long long*>(At[d] + off(b)); };
                    const long long z = Z(0) + Z(1) + Z(2);
                    double v;
                    if constexpr (DIR) {
                        if (more) fetch_dir(gn, b);
                        v = bad ? C : fx_ldexp(z, x);
                    } else {
                        const double hi = __hiloint2double(0x45300000 + X, (int)((unsigned)(z >> 32) ^ 0x80000000u));
                        const double lo = __hiloint2double(0x43300000 + X, (int)(unsigned)z);
                        v = __dadd_rn(__dsub_rn(hi, C), lo);
                    }
                    we[b * TPE] = v;
                    if constexpr (mode_energies(MODE)) energy = fma(ue[b], v, energy);
                }
            }
        }
        if constexpr (mode_energies(MODE)) S.esum[tid] = energy;
        prev = e0;
        buf ^= 1;
        e0 = enext;
    }
    if constexpr (mode_energies(MODE)) {
        __syncthreads();
        flush_energies();
    }
}

}  // namespace

}  // namespace nek

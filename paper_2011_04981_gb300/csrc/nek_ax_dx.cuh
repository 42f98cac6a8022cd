// AX operator in FP64, nx >= 3: the line-pass kernel.
//
// The operator is Section II-B's, Listing 1 of arXiv 2011.04981, per element
//   ur = D_r u, us = D_s u, ut = D_t u             (local_grad3)
//   [wr ws wt] = G [ur us ut]                        (the pointwise g product)
//   w = D_r^T wr + D_s^T ws + D_t^T wt               (local_grad3_t)
// with D_r acting on i, D_s on j and D_t on k of the [k][j][i] block.
//
// GB300 has two FP64 lanes per SM and clock; the contractions alone (12 nx operations a point) kept that pipe busy for
// the whole time of the FP64 form (nx = 8, 8000 elements: 348 us at the pipe's rate, 408 measured).  Its 64 integer
// multiply-adds (IMAD.WIDE) per clock take the contractions instead, in block fixed point per line, with FP64 for G:
//   - a line's values become 58-bit integers at the scale of its largest, a matrix row 58-bit integers at the scale of
//     its absolute sum, each as two 29-bit digits;
//   - the high digits' products and the two cross products are summed exactly in 64 bits; the products of the low digits,
//     each below 2^-58 of the line's bound, are dropped.  The sum is rounded to a double by shifts (dx_ldexp);
//   - D of a symmetric rule satisfies D[n-1-i][n-1-l] = -D[i][l]: with the sums and differences of mirrored points every
//     product serves two outputs.  The kernel checks that of the D it is given and otherwise computes every row.
// A result's error is at most 2^-53 of its size (the final rounding) plus (2 nx + 4) 2^-57 of the line's largest value times
// the row's absolute sum: the values' digits are truncated (2 of these), the matrix's rounded (nx), the low digits'
// products dropped (nx + 1), the cross sums rounded (1).  An exact integer model gives up to 1.4 2^-57 at nx = 8 and 1.7 2^-57
// at 16 (150 lines each, random, nearly equal and smooth).  A chain of nx FP64 multiply-adds has up to nx 2^-53 of the sum of
// the terms' magnitudes; that is less only where D has a zero or small entry at a line's largest value (the zero diagonal of
// a rule: a derivative there is good to 2^-57 of the line, not of its own size), and the sum of the three directions then
// has larger terms from the same line.  Measured against 128-bit arithmetic (2-norm, deformed boxes, random u; FP64 form in
// brackets): nx = 4 1.0e-16 (1.2e-16), 8 0.9e-16 (2.0e-16), 16 1.1e-16 (2.7e-16); smooth u, whose derivatives cancel: nx = 8
// 2.4e-16 (1.8e-15).  Lines that are not finite, or outside 2^+-400, are summed in FP64 as they stand, and every line is if a
// row of D is outside.
//
// Mapping: as k_ax_fx: a thread owns two (or one) of the element's 3 nx^2 lines, holds their digits in registers and writes
// all their outputs; G and the result are point-wise over the same threads.  CTAs are persistent, the next element's
// input is copied to shared memory (cp.async) under the current one's second half, G fetched into L2 during phase 1.
//
// What bounds it (nx = 8, 8000 elements, ncu): the FP64 pipe is 63 % busy with the G product (9 operations a point; 4.5
// clocks, 64 us of the 122), the issue slots 50 %, ALU 52 %; the rest is the latency of the phases between the barriers of
// 8 CTAs an SM.  412 -> 122 us; nx = 5 97 -> 49, 16 5.71 -> 1.64 ms (8000 elements), nx = 4 at 196608 elements 709 -> 503.
// 64 elements at nx = 8 30 -> 6.8 us.
#pragma once

#include "nek_internal.h"
#include "nek_lines.cuh"

namespace nek {

namespace {

// Lines per thread where elements fill the chip, and the resident warps per SM that the register budget is set for.  Two
// lines share the loads of the matrix tables (nx = 8 128 against 141 us, 13 168 against 195, 15 221 against 229); at nx = 16
// the block of 12 warps that would leave is slower (232 against 226).  Warps (us, 8 million points): up to nx = 7 32 (nx = 5
// 277, 288 with 28; 7 285, 291); 8 24 or 28 (233; 254 with 20, 237 with 32); 12, 13 and 15 24 and more alike (336, 327, 424;
// 355, 336, 461 with 20); 9 and 10 277 and 292 with 28, 268 and 287 with 24 (nx = 10 at 4.1 million points 156 with 28, 160
// with 24); 14 and 16 the same from 20 on (shared memory).
constexpr int dx_lpt(int nx) { return nx <= 15 ? 2 : 1; }
constexpr int dx_warps(int nx) { return nx <= 7 ? 32 : nx == 8 || nx == 12 || nx == 13 || nx >= 15 ? 24 : 28; }
constexpr int dx_tpe(int nx, int lpt) { return (3 * nx * nx + lpt - 1) / lpt; }
constexpr int dx_threads(int nx, int epb, int lpt) { return (dx_tpe(nx, lpt) * epb + 31) / 32 * 32; }

// The folded matrix of one phase.  Row i, entry l < ceil(n/2): the integers a_l + a_{n-1-l} (even part, multiplies the sum of
// the mirrored points) and a_l - a_{n-1-l} (odd part, the difference), a the row times 2^(58 - ex), each as two digits.
template <int NX>
struct DxTab {
    static constexpr int HE = (NX + 1) / 2;
    int4 d[NX * HE];  // even high, even low, odd high, odd low
    int ex[NX];       // 2^ex is above the row's absolute sum
};

template <int NX, int EPB>
struct DxSmem {
    static constexpr int NP = FxGrid<NX>::SIZE;
    double U[EPB * NP];
    double A[3][EPB * NP];  // derivatives, then products with G, then the line sums of phase 2
    DxTab<NX> tab[2];  // of D and of its transpose
    double D[NX * NX];
};

// Exponents (unbiased) within which a line's largest magnitude and a matrix row's absolute sum are taken in fixed point: no
// result overflows or underflows.  Lines outside (also infinities, NaNs) are summed in FP64 as they stand.
constexpr int kDxRange = 400;
constexpr int kDxDigit = 29;

__device__ __forceinline__ int dx_high(long long v) { return (int)((v + (1ll << (kDxDigit - 1))) >> kDxDigit); }
__device__ __forceinline__ int dx_low(long long v) { return (int)(v - ((long long)dx_high(v) << kDxDigit)); }

// z 2^x as a double, rounded to nearest (ties away from zero), for x such that nothing overflows or underflows: no FP64
// instruction.
__device__ __forceinline__ double dx_ldexp(long long z, int x)
{
    const int sg = (int)(z >> 32) >> 31;
    const unsigned long long a = (unsigned long long)((z ^ (long long)sg) - (long long)sg);
    const int lz = __clzll((long long)a);
    unsigned long long g;
    asm("shl.b64 %0, %1, %2;" : "=l"(g) : "l"(a), "r"(lz));
    const unsigned long long m = (g >> 11) + ((unsigned)g >> 10 & 1u);  // leading one at bit 52 (53 after a carry)
    const unsigned hi = (unsigned)(m >> 32) + ((unsigned)(1085 + x - lz) << 20);  // the leading one adds 1
    return __hiloint2double((int)((int)(g >> 32) >= 0 ? 0u : hi | ((unsigned)sg & 0x80000000u)), (int)(unsigned)m);
}

// Copies the matrix Dg to D, finds out whether it is symmetric as above, and fills t[0] (M = D) and t[1] (M = D^T), in
// integers (an FP64 chain here would be a third of the time of a call on few elements).  Returns whether a row's absolute
// sum is outside kDxRange; the tables are then not to be used.
template <int NX>
__device__ __forceinline__ bool dx_build(const double* __restrict__ Dg, double* D, DxTab<NX>* t, int tid, int nt, bool& sym)
{
    constexpr int HE = DxTab<NX>::HE, N2 = NX * NX;
    for (int q = tid; q < N2; q += nt) D[q] = Dg[q];
    __syncthreads();
    bool asym = false;
    for (int q = tid; q < N2; q += nt) asym = asym || D[q] != -D[N2 - 1 - q];
    sym = !__syncthreads_or(asym);
    auto entry = [&](int m, int i, int l) { return m ? D[l * NX + i] : D[i * NX + l]; };
    bool bad = false;
    for (int r = tid; r < 2 * NX; r += nt) {
        const int m = r / NX, i = r - m * NX;
        unsigned E = 0u, any = 0u;
        for (int l = 0; l < NX; l++) {
            const double v = entry(m, i, l);
            E = max(E, (unsigned)__double2hiint(v) & 0x7FFFFFFFu);
            any |= (unsigned)__double2loint(v);
        }
        any |= E;
        E >>= 20;
        unsigned sum = 0u;  // above the row's absolute sum, in units of 2^(E - 1043)
        for (int l = 0; l < NX; l++) {
            const unsigned hi = (unsigned)__double2hiint(entry(m, i, l));
            sum += (((hi & 0xFFFFFu) | 0x100000u) >> min(E - (hi >> 20 & 0x7FFu), 31u)) + 1u;
        }
        const int e = any ? (int)E - 1043 + 32 - __clz((int)sum) : 0;
        bad = bad || e < -kDxRange || e > kDxRange;
        t[m].ex[i] = e;
    }
    if (__syncthreads_or(bad)) return true;
    for (int q = tid; q < 2 * NX * HE; q += nt) {
        const int m = q / (NX * HE), p = q - m * NX * HE, i = p / HE, l = p - i * HE;
        const int e = t[m].ex[i];
        auto fixed = [&](double v) {  // v 2^(2 kDxDigit - e) to the nearest integer
            const unsigned hi = (unsigned)__double2hiint(v);
            const unsigned long long mant =
                ((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32) | (unsigned)__double2loint(v);
            const int s = e + 1022 - (int)(hi >> 20 & 0x7FFu);
            const long long f = s > 62 ? 0 : (long long)(((mant << (2 * kDxDigit - 52) >> s) + 1) >> 1);
            return (int)hi < 0 ? -f : f;
        };
        const long long a = fixed(entry(m, i, l)), b = fixed(entry(m, i, NX - 1 - l));
        t[m].d[p] = make_int4(dx_high(a + b), dx_low(a + b), dx_high(a - b), dx_low(a - b));
    }
    return false;
}

// One line pass over LPT lines of NX points: src[q] and dst[q] hold NX values at stride st[q]; sg[q] is the sign bit to
// apply to the input.
template <int NX, bool TRANS, int LPT>
__device__ __forceinline__ void dx_lines(const double* const (&src)[LPT], double* const (&dst)[LPT], const int (&st)[LPT],
                                         const unsigned (&sg)[LPT], const DxTab<NX>& tab, const double* D, bool sym, bool bad)
{
    constexpr int HE = DxTab<NX>::HE, HO = NX / 2;
    constexpr long long kHalf = 1ll << (kDxDigit - 1);
    constexpr unsigned kMask = (1u << kDxDigit) - 1u;
    int sh[LPT][HE], sl[LPT][HE], dh[LPT][HE], dl[LPT][HE], ex[LPT];
    bool slow[LPT];
#pragma unroll
    for (int q = 0; q < LPT; q++) {
        double v[NX];
        unsigned mx = 0u;
#pragma unroll
        for (int l = 0; l < NX; l++) {
            v[l] = src[q][l * st[q]];
            mx = max(mx, (unsigned)__double2hiint(v[l]) & 0x7FFFFFFFu);
        }
        slow[q] = bad;
        if (mx - ((1023u - kDxRange) << 20) >= (2u * kDxRange) << 20) {  // zero, small, large or not finite
            unsigned any = 0u;
#pragma unroll
            for (int l = 0; l < NX; l++)
                any |= ((unsigned)__double2hiint(v[l]) & 0x7FFFFFFFu) | (unsigned)__double2loint(v[l]);
            slow[q] = bad || any != 0u;
            mx = 1023u << 20;
        }
        const unsigned E = mx & 0x7FF00000u;
        ex[q] = (int)(E >> 20) - (1023 + 2 * kDxDigit);
        // |v| as an integer of 58 bits at the scale of the line's largest (truncated), in two digits with v's sign
        auto conv = [&](double x, int& h, int& l) {
            const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
            const unsigned s = (E - (hi & 0x7FF00000u)) >> 20;
            const unsigned mh = (hi & 0x000FFFFFu) | 0x00100000u;
            constexpr int kUp = 2 * kDxDigit - 53;
            const unsigned long long m = ((unsigned long long)__funnelshift_l(lo, mh, kUp) << 32) | (lo << kUp);
            unsigned long long a, b;
            asm("shr.u64 %0, %1, %2;" : "=l"(a) : "l"(m), "r"(s + kDxDigit));
            asm("shr.u64 %0, %1, %2;" : "=l"(b) : "l"(m), "r"(s));
            const int sn = (int)(hi ^ sg[q]) >> 31;
            h = ((int)(unsigned)a ^ sn) - sn;
            l = ((int)((unsigned)b & kMask) ^ sn) - sn;
        };
#pragma unroll
        for (int l = 0; l < HE; l++) {
            const int m = NX - 1 - l;
            int h, o;
            conv(v[l], h, o);
            if (l == m) {
                sh[q][l] = h;
                sl[q][l] = o;
            } else {
                int h2, o2;
                conv(v[m], h2, o2);
                sh[q][l] = h + h2;
                dh[q][l] = h - h2;
                sl[q][l] = o + o2;
                dl[q][l] = o - o2;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < LPT; q++) {
        if (!slow[q] || (q > 0 && src[q] == src[0])) continue;
        double c[NX];
        for (int l = 0; l < NX; l++) {
            const double x = src[q][l * st[q]];
            c[l] = sg[q] ? -x : x;
        }
#pragma unroll 1
        for (int i = 0; i < NX; i++) {
            double s = 0.0;
#pragma unroll 1
            for (int l = 0; l < NX; l++) s = fma(TRANS ? D[l * NX + i] : D[i * NX + l], c[l], s);
            dst[q][i * st[q]] = s;
        }
    }
    auto row = [&](int i, long long (&e)[LPT], long long (&o)[LPT]) {
        long long ah[LPT], ac[LPT], bh[LPT], bc[LPT];
#pragma unroll
        for (int l = 0; l < HE; l++) {
            const int4 t = tab.d[i * HE + l];
#pragma unroll
            for (int q = 0; q < LPT; q++) {
                ah[q] = l == 0 ? (long long)sh[q][0] * t.x : madw(sh[q][l], t.x, ah[q]);
                ac[q] = madw(sl[q][l], t.x, l == 0 ? kHalf : ac[q]);
                ac[q] = madw(sh[q][l], t.y, ac[q]);
                if (l < HO) {
                    bh[q] = l == 0 ? (long long)dh[q][0] * t.z : madw(dh[q][l], t.z, bh[q]);
                    bc[q] = madw(dl[q][l], t.z, l == 0 ? kHalf : bc[q]);
                    bc[q] = madw(dh[q][l], t.w, bc[q]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < LPT; q++) {
            e[q] = ah[q] + (ac[q] >> kDxDigit);
            o[q] = bh[q] + (bc[q] >> kDxDigit);
        }
    };
    if (sym) {
#pragma unroll 1
        for (int i = 0; i < HE; i++) {
            long long e[LPT], o[LPT];
            row(i, e, o);
            const int x1 = tab.ex[i], x2 = tab.ex[NX - 1 - i];
#pragma unroll
            for (int q = 0; q < LPT; q++) {
                if (slow[q]) continue;
                dst[q][i * st[q]] = dx_ldexp(e[q] + o[q], ex[q] + x1);
                if (HE == HO || i < HO) dst[q][(NX - 1 - i) * st[q]] = dx_ldexp(o[q] - e[q], ex[q] + x2);
            }
        }
    } else {
#pragma unroll 1
        for (int i = 0; i < NX; i++) {
            long long e[LPT], o[LPT];
            row(i, e, o);
            const int x = tab.ex[i];
#pragma unroll
            for (int q = 0; q < LPT; q++)
                if (!slow[q]) dst[q][i * st[q]] = dx_ldexp(e[q] + o[q], ex[q] + x);
        }
    }
}

// A thread's lines (line L of an element: direction L / nx^2, line L % nx^2 of it), t the thread's number within its
// element, slot the element's place; a thread whose last line would be past the end repeats its first.
template <int NX, int LPT>
struct DxLines {
    const double *u[LPT], *in[LPT];  // phase 1 and phase 2 inputs
    double* a[LPT];
    int str[LPT];
    unsigned sgn[LPT];

    __device__ __forceinline__ DxLines(double* U, double* A0, int astride, int slot, int t, bool sym)
    {
        using Grid = FxGrid<NX>;
        constexpr int N2 = NX * NX, TPE = dx_tpe(NX, LPT);
#pragma unroll
        for (int q = 0; q < LPT; q++) {
            const int L = t + q * TPE < 3 * N2 ? t + q * TPE : t;
            const int d = L / N2, c = L - d * N2, y = c / NX, x = c - y * NX;
            int base = slot + (d == 0 ? x * Grid::ROW + y * Grid::PLANE : x + y * (d == 1 ? Grid::PLANE : Grid::ROW));
            str[q] = d == 0 ? 1 : d == 1 ? Grid::ROW : Grid::PLANE;
            sgn[q] = 0u;
            if (Grid::REV != 0 && d == 0 && sym && (t / (Grid::REV ? Grid::REV : 1)) & 1) {
                base += NX - 1;
                str[q] = -1;
                sgn[q] = 0x80000000u;
            }
            u[q] = U + base;
            a[q] = A0 + d * astride + base;
            in[q] = a[q];
        }
    }
};

// [wr ws wt] = G [ur us ut] in place on the thread's points t, t + TPE, ... of an element; Ge: its factors.
template <int NX, int TPE>
__device__ __forceinline__ void dx_geom(const double* __restrict__ Ge, double* const (&At)[3], int t)
{
    using Grid = FxGrid<NX>;
    const double2* gp = reinterpret_cast<const double2*>(Ge + 6 * t);
#pragma unroll 3
    for (int p = t; p < NX * NX * NX; p += TPE, gp += 3 * TPE) {
        const int a = Grid::at(p) - Grid::at(t);
        const double2 g01 = __ldg(gp), g23 = __ldg(gp + 1), g45 = __ldg(gp + 2);
        const double ar = At[0][a], as = At[1][a], at = At[2][a];
        At[0][a] = fma(g01.x, ar, fma(g01.y, as, g23.x * at));
        At[1][a] = fma(g01.y, ar, fma(g23.y, as, g45.x * at));
        At[2][a] = fma(g23.x, ar, fma(g45.x, as, g45.y * at));
    }
}

template <int NX, int EPB, int LPT>
constexpr int dx_min_blocks()
{
    const int by_smem = (int)((227 * 1024) / (sizeof(DxSmem<NX, EPB>) + 1024));
    const int by_warps = dx_warps(NX) / (dx_threads(NX, EPB, LPT) / 32);
    const int b = by_smem < by_warps ? by_smem : by_warps;
    return b < 1 ? 1 : b;
}

template <int NX, int EPB, int LPT>
__global__ void __launch_bounds__(dx_threads(NX, EPB, LPT), (dx_min_blocks<NX, EPB, LPT>()))
    k_ax_dx(int64_t nelt, const double* __restrict__ D, const double* __restrict__ G, const double* __restrict__ u,
            double* __restrict__ w)
{
    using Grid = FxGrid<NX>;
    constexpr int NP = Grid::SIZE, N3 = NX * NX * NX;
    constexpr int TPE = dx_tpe(NX, LPT), NT = dx_threads(NX, EPB, LPT);
    constexpr int B = (N3 + TPE - 1) / TPE;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DxSmem<NX, EPB>& S = *reinterpret_cast<DxSmem<NX, EPB>*>(smem_raw);
    const int tid = threadIdx.x, el = tid / TPE, t = tid - el * TPE;
    const int slot = (el < EPB ? el : 0) * NP;
    double* Ut = S.U + slot + Grid::at(t);
    auto off = [&](int b) {
        if constexpr (Grid::ROW == NX && Grid::PAD == 0)
            return b * TPE;
        else
            return Grid::at(t + b * TPE) - Grid::at(t);
    };
    auto has = [&](int b) { return b < B - 1 || t + b * TPE < N3; };
    auto fetch = [&](int64_t g0) {
        if (el < EPB && g0 + el < nelt) {
            const double* src = u + (g0 + el) * (int64_t)N3 + t;
#pragma unroll
            for (int b = 0; b < B; b++)
                if (has(b)) cp_async8(Ut + off(b), src + b * TPE);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int64_t step = (int64_t)gridDim.x * EPB;
    int64_t e0 = (int64_t)blockIdx.x * EPB;
    fetch(e0);

    // ---- the matrix tables, once per CTA
    bool sym;
    const bool bad = dx_build<NX>(D, S.D, S.tab, tid, NT, sym);

    DxLines<NX, LPT> ln(S.U, S.A[0], EPB * NP, slot, t, sym);
    double* At[3];
#pragma unroll
    for (int d = 0; d < 3; d++) At[d] = S.A[d] + slot + Grid::at(t);

    for (; e0 < nelt; e0 += step) {
        const int ne = static_cast<int>(nelt - e0 < EPB ? nelt - e0 : EPB);
        const bool active = el < ne;
        const int64_t ef = (e0 + el) * (int64_t)N3;
        if (tid == 0)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(G + e0 * N3 * 6), "r"((unsigned)(ne * N3 * 48))
                         : "memory");
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (active) dx_lines<NX, false, LPT>(ln.u, ln.a, ln.str, ln.sgn, S.tab[0], S.D, sym, bad);
        __syncthreads();
        if (e0 + step < nelt) fetch(e0 + step);  // U is free: every line has been read
        if (active) dx_geom<NX, TPE>(G + ef * 6, At, t);
        __syncthreads();
        if (active) dx_lines<NX, true, LPT>(ln.in, ln.a, ln.str, ln.sgn, S.tab[1], S.D, sym, bad);
        __syncthreads();
        if (active) {
            double* we = w + ef + t;
#pragma unroll
            for (int b = 0; b < B; b++)
                if (has(b)) we[b * TPE] = (At[0][off(b)] + At[1][off(b)]) + At[2][off(b)];
        }
    }
}

// Elements of a CTA that k_ax_dx holds at a time when EPB are asked for (the results do not depend on it): packing pays
// where one element's lines do not fill warps; from nx = 9 on it measured slower (nx = 9, 8000 elements: 202, 249 and 310
// us with 1, 2 and 4) and one is held.
constexpr int dx_conc(int nx, int epb) { return nx >= 9 ? 1 : epb; }

// The fastest of 1, 2 and 4 (8000 elements, us: nx = 5 49 with 4, 62 with 1; 7 111 with 2, 123 with 1; 8 122 with 1, 146
// with 2).
constexpr int dx_default_epb(int nx) { return nx == 3 || nx == 7 ? 2 : nx <= 5 ? 4 : 1; }

template <int NX, int EPB, int LPT>
nek_status configure_dx()
{
    constexpr size_t smem = sizeof(DxSmem<NX, EPB>);
    static_assert(smem <= 227 * 1024 && dx_threads(NX, EPB, LPT) <= 1024, "fits an SM");
    static std::atomic<uint64_t> configured{0};
    return ensure_dyn_smem(k_ax_dx<NX, EPB, LPT>, smem, configured);
}

template <int NX, int EPB, int LPT>
nek_status launch_dx_kernel(int64_t nelt, const double* D, const double* G, const double* u, double* w, cudaStream_t s)
{
    constexpr size_t smem = sizeof(DxSmem<NX, EPB>);
    nek_status st = configure_dx<NX, EPB, LPT>();
    // and the form of few elements: a solve whose launches shrink to it may first do so inside a graph's capture
    if (st == NEK_OK) st = configure_dx<NX, 1, 1>();
    if (st != NEK_OK) return st;
    const int64_t groups = (nelt + EPB - 1) / EPB, resident = kSMs * dx_min_blocks<NX, EPB, LPT>();
    k_ax_dx<NX, EPB, LPT><<<(unsigned)(groups < resident ? groups : resident), dx_threads(NX, EPB, LPT), smem, s>>>(
        nelt, D, G, u, w);
    return check_launch();
}

// epb: elements per CTA asked for (0: the default, dx_default_epb).  With no more elements than SMs there is one to a CTA
// whatever is asked for, and a thread takes one line: twice the warps on each element (nx = 8, 64 elements: 6.8 against 9.3
// us).  The results depend on neither.
template <int NX>
nek_status launch_ax_dx(int epb, int64_t nelt, const double* D, const double* G, const double* u, double* w, cudaStream_t s)
{
    constexpr int L = dx_lpt(NX);
    if (nelt <= kSMs) return launch_dx_kernel<NX, 1, 1>(nelt, D, G, u, w, s);
    if (epb <= 0) epb = dx_default_epb(NX);
    if ((nelt + epb - 1) / epb > 0x7fffffff) return NEK_ERR_TOO_LARGE;
    if (epb == 1) return launch_dx_kernel<NX, 1, L>(nelt, D, G, u, w, s);
    if (epb == 2) return launch_dx_kernel<NX, dx_conc(NX, 2), L>(nelt, D, G, u, w, s);
    return launch_dx_kernel<NX, dx_conc(NX, 4), L>(nelt, D, G, u, w, s);
}

}  // namespace

// Per-nx launchers (nek_ax_dx_<group>.cu: a = nx 3-7, b = 8-11, c = 12-16).
nek_status launch_ax_dx_a(int nx, int epb, int64_t nelt, const double* D, const double* G, const double* u, double* w,
                          cudaStream_t s);
nek_status launch_ax_dx_b(int nx, int epb, int64_t nelt, const double* D, const double* G, const double* u, double* w,
                          cudaStream_t s);
nek_status launch_ax_dx_c(int nx, int epb, int64_t nelt, const double* D, const double* G, const double* u, double* w,
                          cudaStream_t s);

}  // namespace nek

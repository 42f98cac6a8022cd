// Geometric factors of trilinear hexahedra at the GLL nodes (set-up kernel).
//
// For element corners X_q (q = di + 2dj + 4dk) the map is
// x(r,s,t) = sum_q X_q (1 + sr r)(1 + ss s)(1 + st t)/8 with s* = +-1.  Its
// columns x_r, x_s, x_t give |J| = x_r . (x_s x x_t) and the contravariant
// gradients grad r = (x_s x x_t)/|J| (cyclically), so
// G_ab = rho_i rho_j rho_k |J| grad r_a . grad r_b, stored (rr,rs,rt,ss,st,tt).
//
// The kernel is bound by the FP64 pipe (2 operations a clock and SM), so it is written for few of them.  In monomials,
// x = sum m_abc r^a s^b t^c (a, b, c = 0, 1).  Along a line of points in r, x_r is constant, x_s and x_t are linear, hence
// so are x_t x x_r and x_r x x_s: a thread forms their coefficients once for its line, and a point costs 21 operations up
// to the three products and |J| instead of 99 (72 of them for the columns from the corners), 18 for the dot products and
// a division.  24^3 elements at nx = 10: 1.6 ms, 4.1 before; the FP64 pipe is 92 % busy.  (x_s x x_t and |J| as
// quadratics in r saved three more operations, and cost accuracy where |J| is small.)
#include <algorithm>

#include "nek_internal.h"

namespace nek {

struct GllParams {
    double xi[kMaxNx];
    double rho[kMaxNx];
};

namespace {

constexpr int kGeomThreads = 128, kGeomElems = 32;  // at most, in shared memory

__device__ __forceinline__ void cross(const double (&u)[3], const double (&v)[3], double (&w)[3])
{
    w[0] = u[1] * v[2] - u[2] * v[1];
    w[1] = u[2] * v[0] - u[0] * v[2];
    w[2] = u[0] * v[1] - u[1] * v[0];
}
__device__ __forceinline__ double dot(const double (&u)[3], const double (&v)[3])
{
    return u[0] * v[0] + u[1] * v[1] + u[2] * v[2];
}

}  // namespace

// A block takes eb elements at a time (gridDim.y blocks share them), a thread the ns-th part of a line (fixed j, k) of one.
__global__ void __launch_bounds__(kGeomThreads) k_geom(int64_t nelt, int nx, int eb, int ns, GllParams gp,
                                                       const double* __restrict__ corners, double* __restrict__ G)
{
    __shared__ double sm[kGeomElems][8][3];  // m_abc at a + 2 b + 4 c
    const int n2 = nx * nx;
    for (int64_t e0 = (int64_t)blockIdx.x * eb; e0 < nelt; e0 += (int64_t)gridDim.x * eb) {
        const int ne = static_cast<int>(nelt - e0 < eb ? nelt - e0 : eb);
        __syncthreads();
        for (int q = threadIdx.x; q < 3 * ne; q += kGeomThreads) {
            const int e = q / 3, d = q - 3 * e;
            double v[8];
#pragma unroll
            for (int c = 0; c < 8; c++) v[c] = 0.125 * corners[(e0 + e) * 24 + 3 * c + d];
#pragma unroll
            for (int bit = 1; bit < 8; bit <<= 1)
#pragma unroll
                for (int c = 0; c < 8; c++)
                    if (!(c & bit)) {
                        const double lo = v[c], hi = v[c | bit];
                        v[c] = lo + hi;
                        v[c | bit] = hi - lo;
                    }
#pragma unroll
            for (int c = 0; c < 8; c++) sm[e][c][d] = v[c];
        }
        __syncthreads();
        for (int q = blockIdx.y * kGeomThreads + threadIdx.x; q < ne * n2 * ns; q += kGeomThreads * gridDim.y) {
            const int part = q / (ne * n2), ql = q - part * (ne * n2);
            const int e = ql / n2, l = ql - e * n2, k = l / nx, j = l - k * nx;
            const int len = (nx + ns - 1) / ns, i0 = part * len, i1 = min(nx, i0 + len);
            const double s = gp.xi[j], t = gp.xi[k];
            const double(*m)[3] = sm[e];
            // x_r = a, x_s = b0 + r b1, x_t = c0 + r c1
            double a[3], b0[3], b1[3], c0[3], c1[3];
#pragma unroll
            for (int d = 0; d < 3; d++) {
                b0[d] = fma(t, m[6][d], m[2][d]);
                b1[d] = fma(t, m[7][d], m[3][d]);
                c0[d] = fma(s, m[6][d], m[4][d]);
                c1[d] = fma(s, m[7][d], m[5][d]);
                a[d] = fma(s, b1[d], fma(t, m[5][d], m[1][d]));
            }
            double q0[3], q1[3], h0[3], h1[3];
            cross(c0, a, q0);  // x_t x x_r = q0 + r q1
            cross(c1, a, q1);
            cross(a, b0, h0);  // x_r x x_s = h0 + r h1
            cross(a, b1, h1);
            const double rjk = gp.rho[j] * gp.rho[k];
            double* g = G + (((e0 + e) * (int64_t)n2 + l) * nx + i0) * 6;
            for (int i = i0; i < i1; i++, g += 6) {
                const double r = gp.xi[i];
                double b[3], c[3], bc[3], ca[3], ab[3];
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    b[d] = fma(r, b1[d], b0[d]);
                    c[d] = fma(r, c1[d], c0[d]);
                    ca[d] = fma(r, q1[d], q0[d]);
                    ab[d] = fma(r, h1[d], h0[d]);
                }
                cross(b, c, bc);
                const double det = dot(a, bc);
                // G_ab = W |J| (v_a/|J|).(v_b/|J|) = W (v_a . v_b) / |J|
                const double wq = gp.rho[i] * rjk / det;
                double2* o = reinterpret_cast<double2*>(g);
                o[0] = make_double2(wq * dot(bc, bc), wq * dot(bc, ca));
                o[1] = make_double2(wq * dot(bc, ab), wq * dot(ca, ca));
                o[2] = make_double2(wq * dot(ca, ab), wq * dot(ab, ab));
            }
        }
    }
}

}  // namespace nek

using namespace nek;

extern "C" nek_status nek_geom(int64_t nelt, int nx, const double* corners, double* G, void* stream)
{
    if (nx < kMinNx || nx > kMaxNx) return NEK_ERR_UNSUPPORTED_NX;
    if (nelt < 0) return NEK_ERR_INVALID_ARG;
    if (nelt == 0) return NEK_OK;
    if (!corners || !G || !is_aligned(corners, 8) || !is_aligned(G, 16)) return NEK_ERR_INVALID_ARG;
    GllParams gp;
    gll_host(nx, gp.xi, gp.rho, nullptr);
    // About two lines a thread and step, as many blocks as fit on the chip; fewer elements a block where that would leave
    // SMs idle.  Lines in parts where one element leaves threads idle, and, up to half as many elements as SMs, until
    // there is a thread for each on every SM; an element over several blocks where that makes more than one SM for it
    // (one SM's FP64 pipe: nx = 16 needs 69 us for an element, 13.5 when a thread took one point; now 1 element 6.7 us, 64
    // elements 36; nx = 10 6.4 and 15, 23.9 and 24 in one block an element).  More blocks or parts from 76 elements on
    // are slower (100 elements of nx = 8 13.3 us with parts, 12.6 without).  The values do not depend on any of it.
    const int n2 = nx * nx;
    int eb = n2 >= 2 * kGeomThreads ? 1 : std::min(kGeomElems, 2 * kGeomThreads / n2);
    eb = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(eb, nelt / 152)));
    int ns = kGeomThreads / (eb * n2);
    if (nelt <= 76) ns = std::max(ns, 152 * kGeomThreads / (static_cast<int>(nelt) * n2));
    ns = std::max(1, std::min(nx, ns));
    const int64_t nb = (nelt + eb - 1) / eb;
    const int parts = static_cast<int>(
        std::max<int64_t>(1, std::min<int64_t>((eb * n2 * ns + kGeomThreads - 1) / kGeomThreads, 2 * 152 / nb)));
    const dim3 grid(static_cast<unsigned>(nb < 152 * 8 ? nb : 152 * 8), static_cast<unsigned>(parts));
    k_geom<<<grid, kGeomThreads, 0, static_cast<cudaStream_t>(stream)>>>(nelt, nx, eb, ns, gp, corners, G);
    return check_launch();
}

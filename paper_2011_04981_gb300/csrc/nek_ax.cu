// AX operator, FP64 (Section II-B, Listing 1 of arXiv 2011.04981): the dispatch over nx, the C entry point, and the kernel
// of nx = 2.  nx >= 3 runs the line-pass kernel of nek_ax_dx.cuh.
//
// nx = 2: a CTA owns EPB elements; thread (e, i, j) keeps the k-line u(i,j,:) and the t-results wt(i,j,:) in
// registers and walks the k planes.  The u block of every element is staged in shared memory once (one coalesced read
// of u: the FPGA design's single read of every grid point of u becomes one pass through HBM here) so that the r- and
// s-contractions read it from shared memory in their own order, which is what the per-matmul reorder buffers of the FPGA
// design (Section III) achieve.  ws goes to shared memory as it is produced; wr is kept in registers until every
// thread has finished reading u, then overwrites the u block.  G is streamed from HBM exactly once, w written exactly once.
// Lines of two points are too short for the line passes: 196608 elements take 72 us here, 86 in k_ax_dx; the latter
// is faster from nx = 3 on (168 against 261 us).
#include <algorithm>

#include "nek_ax_dx.cuh"
#include "nek_internal.h"

namespace nek {

namespace {

template <int NX, int EPB>
constexpr size_t ax_smem_bytes()
{
    return sizeof(double) * (size_t)(NX * NX + 2 * EPB * NX * NX * NX + 1);
}

template <int NX, int EPB>
__global__ void __launch_bounds__(NX* NX* EPB) k_ax_fp64(int64_t nelt, const double* __restrict__ D,
                                                          const double* __restrict__ G,
                                                          const double* __restrict__ u, double* __restrict__ w)
{
    constexpr int N2 = NX * NX, N3 = NX * NX * NX, NT = N2 * EPB;
    constexpr int DPAD = (N2 + 1) & ~1;  // keep the element blocks 16-byte aligned
    extern __shared__ double smem[];
    double* sD = smem;
    double* sA = smem + DPAD;     // u, then wr   [EPB][N3]
    double* sB = sA + EPB * N3;   // ws           [EPB][N3]

    const int tid = threadIdx.x;
    const int64_t e0 = (int64_t)blockIdx.x * EPB;
    const int ne = static_cast<int>(nelt - e0 < EPB ? nelt - e0 : EPB);

    for (int q = tid; q < N2; q += NT) sD[q] = D[q];
    if ((reinterpret_cast<uintptr_t>(u + e0 * N3) & 15) == 0) {  // 16-byte aligned block start: vector loads
        const double2* src = reinterpret_cast<const double2*>(u + e0 * N3);
        double2* dst = reinterpret_cast<double2*>(sA);
        const int nv = (ne * N3) / 2;
        for (int q = tid; q < nv; q += NT) dst[q] = __ldg(src + q);
        if ((ne * N3) & 1) {
            if (tid == 0) sA[ne * N3 - 1] = __ldg(u + e0 * N3 + ne * N3 - 1);
        }
    } else {
        const double* src = u + e0 * N3;
        for (int q = tid; q < ne * N3; q += NT) sA[q] = __ldg(src + q);
    }
    __syncthreads();

    const int el = tid / N2;
    const int q2 = tid - el * N2;
    const int i = q2 % NX, j = q2 / NX;
    const bool active = el < ne;
    double* ue = sA + el * N3;
    double* se = sB + el * N3;

    double ul[NX], wr[NX], wt[NX];
    if (active) {
#pragma unroll
        for (int l = 0; l < NX; l++) ul[l] = ue[i + NX * (j + NX * l)];
        const double* Ge = G + (e0 + el) * (int64_t)N3 * 6;
#pragma unroll
        for (int k = 0; k < NX; k++) {
            const int p = i + NX * (j + NX * k);
            double ar = 0.0, as = 0.0, at = 0.0;
#pragma unroll
            for (int l = 0; l < NX; l++) {
                ar = fma(sD[i * NX + l], ue[l + NX * (j + NX * k)], ar);
                as = fma(sD[j * NX + l], ue[i + NX * (l + NX * k)], as);
                at = fma(sD[k * NX + l], ul[l], at);
            }
            const double2* g2 = reinterpret_cast<const double2*>(Ge + 6 * p);
            const double2 g01 = __ldg(g2), g23 = __ldg(g2 + 1), g45 = __ldg(g2 + 2);
            wr[k] = fma(g01.x, ar, fma(g01.y, as, g23.x * at));
            se[p] = fma(g01.y, ar, fma(g23.y, as, g45.x * at));
            wt[k] = fma(g23.x, ar, fma(g45.x, as, g45.y * at));
        }
    }
    __syncthreads();  // every thread is done reading u
    if (active) {
#pragma unroll
        for (int k = 0; k < NX; k++) ue[i + NX * (j + NX * k)] = wr[k];
    }
    __syncthreads();
    if (active) {
        double* we = w + (e0 + el) * (int64_t)N3;
#pragma unroll
        for (int k = 0; k < NX; k++) {
            double s = 0.0;
#pragma unroll
            for (int l = 0; l < NX; l++) {
                s = fma(sD[l * NX + i], ue[l + NX * (j + NX * k)], s);
                s = fma(sD[l * NX + j], se[i + NX * (l + NX * k)], s);
                s = fma(sD[l * NX + k], wt[l], s);
            }
            we[i + NX * (j + NX * k)] = s;
        }
    }
}

template <int NX, int EPB>
nek_status launch_ax_variant(int64_t nelt, const double* D, const double* G, const double* u, double* w,
                             cudaStream_t s)
{
    constexpr size_t smem = ax_smem_bytes<NX, EPB>();
    static std::atomic<uint64_t> configured{0};
    nek_status st = ensure_dyn_smem(k_ax_fp64<NX, EPB>, smem, configured);
    if (st != NEK_OK) return st;
    const int64_t blocks = (nelt + EPB - 1) / EPB;
    if (blocks > 0x7fffffff) return NEK_ERR_TOO_LARGE;
    k_ax_fp64<NX, EPB><<<(unsigned)blocks, NX * NX * EPB, smem, s>>>(nelt, D, G, u, w);
    return check_launch();
}

// The elements-per-CTA counts that are accepted: 1, 2 and 4; at nx = 16 1 and 2 (the set does not depend on the kernels
// that run: see ax_fp64_form for which of them differ).
constexpr bool ax_fits(int nx, int epb)
{
    return (epb == 1 || epb == 2 || epb == 4) && nx * nx * epb <= 1024 &&
           (nx * nx + 2 * epb * nx * nx * nx + 1) * 8 <= 227 * 1024;
}

}  // namespace

nek_status launch_ax_fp64_epb(int epb, int64_t nelt, int nx, const double* D, const double* G, const double* u,
                              double* w, cudaStream_t s)
{
    if (nx < kMinNx || nx > kMaxNx) return NEK_ERR_UNSUPPORTED_NX;
    if (epb > 0 && !ax_fits(nx, epb)) return NEK_ERR_INVALID_ARG;
    if (nx == 2) {
        switch (epb) {
            case 1: return launch_ax_variant<2, 1>(nelt, D, G, u, w, s);
            case 2: return launch_ax_variant<2, 2>(nelt, D, G, u, w, s);
            case 4: return launch_ax_variant<2, 4>(nelt, D, G, u, w, s);
            default: return launch_ax_variant<2, 32>(nelt, D, G, u, w, s);
        }
    }
    if (nx <= 7) return launch_ax_dx_a(nx, epb, nelt, D, G, u, w, s);
    if (nx <= 11) return launch_ax_dx_b(nx, epb, nelt, D, G, u, w, s);
    return launch_ax_dx_c(nx, epb, nelt, D, G, u, w, s);
}

bool ax_fp64_epb_fits(int nx, int epb) { return nx >= kMinNx && nx <= kMaxNx && ax_fits(nx, epb); }

int ax_fp64_default_epb(int nx) { return nx == 2 ? 0 : dx_default_epb(nx); }

int ax_fp64_form(int64_t nelt, int nx, int epb)
{
    if (nx == 2) return epb > 0 ? epb : 32;
    return nelt <= kSMs ? 0 : dx_conc(nx, epb > 0 ? epb : dx_default_epb(nx));
}

nek_status launch_ax_fp64(int64_t nelt, int nx, const double* D, const double* G, const double* u, double* w,
                          cudaStream_t s)
{
    return launch_ax_fp64_epb(tuned_epb(NEK_AX_FP64, nx), nelt, nx, D, G, u, w, s);
}

}  // namespace nek

using namespace nek;

extern "C" nek_status nek_ax(int64_t nelt, int nx, const double* D, const double* G, const double* u, double* w,
                             void* stream)
{
    if (nx < kMinNx || nx > kMaxNx) return NEK_ERR_UNSUPPORTED_NX;
    if (nelt < 0) return NEK_ERR_INVALID_ARG;
    if (nelt == 0) return NEK_OK;
    if (!D || !G || !u || !w) return NEK_ERR_INVALID_ARG;
    if (!is_aligned(D, 8) || !is_aligned(G, 16) || !is_aligned(u, 8) || !is_aligned(w, 8))
        return NEK_ERR_INVALID_ARG;
    const size_t bytes = sizeof(double) * (size_t)nelt * nx * nx * nx;
    if (ranges_overlap(u, bytes, w, bytes)) return NEK_ERR_INVALID_ARG;
    return launch_ax_fp64(nelt, nx, D, G, u, w, static_cast<cudaStream_t>(stream));
}

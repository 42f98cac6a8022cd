// FP64 AX launchers for nx = 12 - 16 (kernel in nek_ax_dx.cuh).
#include "nek_ax_dx.cuh"

namespace nek {

nek_status launch_ax_dx_c(int nx, int epb, int64_t nelt, const double* D, const double* G, const double* u, double* w,
                          cudaStream_t s)
{
    switch (nx) {
        case 12: return launch_ax_dx<12>(epb, nelt, D, G, u, w, s);
        case 13: return launch_ax_dx<13>(epb, nelt, D, G, u, w, s);
        case 14: return launch_ax_dx<14>(epb, nelt, D, G, u, w, s);
        case 15: return launch_ax_dx<15>(epb, nelt, D, G, u, w, s);
        case 16: return launch_ax_dx<16>(epb, nelt, D, G, u, w, s);
        default: return NEK_ERR_UNSUPPORTED_NX;
    }
}

}  // namespace nek

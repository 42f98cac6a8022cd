// FP64 AX launchers for nx = 8 - 11 (kernel in nek_ax_dx.cuh).
#include "nek_ax_dx.cuh"

namespace nek {

nek_status launch_ax_dx_b(int nx, int epb, int64_t nelt, const double* D, const double* G, const double* u, double* w,
                          cudaStream_t s)
{
    switch (nx) {
        case 8: return launch_ax_dx<8>(epb, nelt, D, G, u, w, s);
        case 9: return launch_ax_dx<9>(epb, nelt, D, G, u, w, s);
        case 10: return launch_ax_dx<10>(epb, nelt, D, G, u, w, s);
        case 11: return launch_ax_dx<11>(epb, nelt, D, G, u, w, s);
        default: return NEK_ERR_UNSUPPORTED_NX;
    }
}

}  // namespace nek

// FP64 AX launchers for nx = 3 - 7 (kernel in nek_ax_dx.cuh).
#include "nek_ax_dx.cuh"

namespace nek {

nek_status launch_ax_dx_a(int nx, int epb, int64_t nelt, const double* D, const double* G, const double* u, double* w,
                          cudaStream_t s)
{
    switch (nx) {
        case 3: return launch_ax_dx<3>(epb, nelt, D, G, u, w, s);
        case 4: return launch_ax_dx<4>(epb, nelt, D, G, u, w, s);
        case 5: return launch_ax_dx<5>(epb, nelt, D, G, u, w, s);
        case 6: return launch_ax_dx<6>(epb, nelt, D, G, u, w, s);
        case 7: return launch_ax_dx<7>(epb, nelt, D, G, u, w, s);
        default: return NEK_ERR_UNSUPPORTED_NX;
    }
}

}  // namespace nek

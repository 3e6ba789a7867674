// Instantiations of the fused stencil / Chebyshev-step kernels (see stencil_impl.cuh)
// for one element type per translation unit, so the variants compile in parallel.
#include "stencil_brick.cuh"

namespace sdft {

template <>
void launch_cheb_step<double2>(sdft_ctx* c, int kpt, const double2* Y, const double2* Yprev, double2* Ynext, int ncolE,
                               const double* V, const double2* kbC, double alpha, double beta, double shift,
                               bool with_kinetic) {
    // us per step between events (column tile -> brick): 24^3 x 8 210 -> 33, 36^3 x 24 570 -> 255, 48^3 x 24 833 -> 550
    if (brick_ok<double2, 4>(c, ncolE) && V != nullptr) {
        launch_brick<double2, true, 4, 2>(c, kpt, Y, Yprev, Ynext, ncolE, V, kbC, alpha, beta, shift, with_kinetic, true);
        return;
    }
    launch_variant<double2, true, 32, 8, 2, 1, 3>(c, kpt, Y, Yprev, Ynext, ncolE, V, kbC, alpha, beta, shift, with_kinetic,
                                              true);
}

template <>
void launch_kb_project<double2>(sdft_ctx* c, int kpt, const double2* Y, double2* C, int ncolE) {
    launch_project_impl<double2>(c, kpt, Y, C, ncolE);
}

}  // namespace sdft

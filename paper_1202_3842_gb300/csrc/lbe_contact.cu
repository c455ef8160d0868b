// K2 launchers (contact values); the kernel is in lbe_contact.cuh.
#include "lbe_contact.cuh"

namespace lbe {

cudaError_t launch_contact_tma(bool fp64, const ContactLaunch &L, cudaStream_t st) {
    return fp64 ? dispatch_m<double, 0>(L, st) : dispatch_m<float, 0>(L, st);
}

void contact_box(bool fp64, int M, int RB, int *bx, int *by) {
    const int A = fp64 ? 2 : 4, nx = fp64 ? 1 : 2;  // ContactTile
    *bx = 32 + 2 * ((RB + A - 1) / A * A);
    *by = CT_THREADS * nx / 32 + 2 * RB;
    (void)M;
}

}  // namespace lbe

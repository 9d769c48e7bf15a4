// Tetrahedron kernels with plane-major inputs and outputs straight from and to global
// memory, every precision form.
#include "fe_inst.cuh"
#include "fe_plane.cuh"
namespace fe {
const void *kernel_plane_tet(int kind, int prec, int quad, int cpq, int outl) {
    FE_PLANE6(FE_PLANE_CASE, TET, FP64, Q_TET1)
    FE_PLANE6(FE_PLANE_CASE, TET, FP64, Q_TET4)
    FE_PLANE6(FE_PLANE_CASE, TET, MIXED, Q_TET1)
    FE_PLANE6(FE_PLANE_CASE, TET, MIXED, Q_TET4)
    FE_PLANE6(FE_PLANE_CASE, TET, DWORD, Q_TET1)
    FE_PLANE6(FE_PLANE_CASE, TET, DWORD, Q_TET4)
    return nullptr;
}
}  // namespace fe

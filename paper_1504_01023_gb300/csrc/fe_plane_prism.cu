// Prism kernels with plane-major inputs and outputs straight from and to global
// memory, every precision form.
#include "fe_inst.cuh"
#include "fe_plane.cuh"
namespace fe {
const void *kernel_plane_prism(int kind, int prec, int quad, int cpq, int outl) {
    FE_PLANE6(FE_PLANE_PAIR_CASE, PRISM, FP64, Q_PRISM6)
    FE_PLANE6(FE_PLANE_CASE, PRISM, MIXED, Q_PRISM6)
    FE_PLANE6(FE_PLANE_CASE, PRISM, DWORD, Q_PRISM6)
    return nullptr;
}
}  // namespace fe

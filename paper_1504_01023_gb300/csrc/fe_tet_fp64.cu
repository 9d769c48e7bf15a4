// Tetrahedron kernels, FP64 form.
#include "fe_inst.cuh"
namespace fe {
const void *kernel_tet_fp64(int kind, int quad, int cpq, int inl, int outl) {
    if (inl == INDEXED) return kernel_tet_fp64_idx(kind, quad, cpq, outl);
    if (quad == Q_TET1) { FE_ALL16(FE_F64T_CASE, TET, FP64, Q_TET1) FE_PK8(FE_F64T_CASE, TET, FP64, Q_TET1) FE_FN2(FE_F64T_CASE, 0, TET, FP64, Q_TET1) FE_FN2(FE_F64T_CASE, 1, TET, FP64, Q_TET1) }
    if (quad == Q_TET4) { FE_ALL16(FE_F64T_CASE, TET, FP64, Q_TET4) FE_PK8(FE_F64T_CASE, TET, FP64, Q_TET4) FE_FN2(FE_F64T_CASE, 0, TET, FP64, Q_TET4) FE_FN2(FE_F64T_CASE, 1, TET, FP64, Q_TET4) }
    return nullptr;
}

// The tile kernel for the element-contiguous sets that stream_kernel_f64t takes, for
// host memory written in place (see launch_set).
const void *kernel_tet_fp64_tile(int kind, int quad, int cpq) {
#define FE_F64_TILE(KD, QD, CP) \
    if (kind == KD && quad == QD && cpq == CP) return reinterpret_cast<const void *>(&elem_kernel_f64t<KD, QD, CP, AOS, AOS>);
    FE_F64_TILE(GENERIC, Q_TET1, 0) FE_F64_TILE(GENERIC, Q_TET4, 0) FE_F64_TILE(POISSON, Q_TET1, 0)
    FE_F64_TILE(POISSON, Q_TET4, 0) FE_F64_TILE(POISSON, Q_TET1, 1) FE_F64_TILE(POISSON, Q_TET4, 1)
#undef FE_F64_TILE
    return nullptr;
}
}  // namespace fe

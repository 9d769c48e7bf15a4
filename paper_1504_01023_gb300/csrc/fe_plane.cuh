// Plane-major inputs and outputs: one element per thread straight between global
// memory and registers.
#pragma once
#include "fe_kernels.cuh"

namespace fe {

// Plane values through the read-only path (read again by forms that scan the
// coefficients first: the second read hits L1).
template <class T> struct PlaneSrc {
    const T *base;
    int64_t stride;
    __device__ __forceinline__ T operator()(int j) const { return __ldg(base + j * stride); }
};

// Scalar j of a warp's 32 elements is one contiguous run of its plane, so loads and
// stores are coalesced whatever the planes' alignment and pitch, every load of a
// thread is in flight at once and no block barrier separates them from the
// arithmetic. skip_mod as for elem_tiles: tiles of blockDim elements.
template <int ET, int KIND, int PREC, int QUAD, int CPQ, int OUTL>
__device__ __forceinline__ void plane_elems(const ElemParams &p, const CoefFn *fn) {
    using CF = ElemCfg<ET, KIND, PREC, QUAD, CPQ>;
    using CT = typename CF::CT;
    constexpr int NS = CF::NS, NX = CF::NX, NA = CF::NA, NC = CF::NC;
    // coefficient planes up to 80 bytes per element are read ahead into registers
    constexpr bool kCoefRegs = NC * sizeof(CT) <= 80;
    const CT *C = static_cast<const CT *>(p.C);
    CT *Aout = static_cast<CT *>(p.A);
    CT *Bout = static_cast<CT *>(p.B);
    grid_wait();
    if (PREC != FP64) grid_trigger();
    const int64_t ntiles = (p.n + blockDim.x - 1) / blockDim.x;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        if (p.skip_mod > 0 && tile % p.skip_mod == 0) {   // injected fault: no load, no store
            if (threadIdx.x == 0) atomicOr(p.status, ST_SKIPPED_TILES);
            continue;
        }
        const int64_t e = tile * blockDim.x + threadIdx.x;
        const bool active = e < p.n;
        bool poor = false;
        if (active) {
            double xr[NX];
#pragma unroll
            for (int j = 0; j < NX; ++j) xr[j] = ld_stream(p.X + j * p.xs + e);
            CT A[NA], b[NS];
            uint8_t fl;
            if constexpr (kCoefRegs) {
                CT cr[NC];
#pragma unroll
                for (int j = 0; j < NC; ++j) cr[j] = ld_stream(C + j * p.cs + e);
                fl = run_elem<ET, KIND, PREC, QUAD, CPQ>(RegSrc<double>{xr}, RegSrc<CT>{cr}, fn, A, b, poor);
            } else {
                fl = run_elem<ET, KIND, PREC, QUAD, CPQ>(RegSrc<double>{xr}, PlaneSrc<CT>{C + e, p.cs}, fn, A, b, poor);
            }
            if (PREC != FP64 && poor) fl |= 1;
            if (p.flags) p.flags[e] = fl;
#pragma unroll
            for (int r = 0; r < NS; ++r)
#pragma unroll
                for (int s = out_packed(OUTL) ? r : 0; s < NS; ++s) {
                    const int ko = out_packed(OUTL) ? packed_index(NS, r, s) : r * NS + s;
                    st_stream(Aout + ko * p.os + e, A[r * NS + s]);
                }
#pragma unroll
            for (int k = 0; k < NS; ++k) st_stream(Bout + k * p.os + e, b[k]);
        }
        if (PREC != FP64) append_fixup(p, active && poor, e);
    }
}

template <int ET, int KIND, int PREC, int QUAD, int CPQ, int OUTL>
__global__ void __launch_bounds__(ET == TET && PREC != DWORD ? 512 : 256)
    plane_kernel(const ElemParams p, const __grid_constant__ TmaMaps, const __grid_constant__ CoefFn fn) {
    plane_elems<ET, KIND, PREC, QUAD, CPQ, OUTL>(p, &fn);
}

// FP64 prisms: two threads per element in block fixed point (PrismFx), bound as
// pair_kernel_f64 by the latency of its chains; both threads read the coordinate
// planes (one sector for the pair), each its level's coefficients and writes its half
// of A^e and b^e. Against the tensor-copied tiles of one thread in doubles, us:
// 300,000 per point 845 / 248, per element 860 / 226, Laplace 311 / 116; 20,000 per
// point 89 / 33, Laplace 35 / 19; 200,000 per point in pinned host memory 1,228 /
// 1,120. Generic kind: 60 values of dynamic shared memory per thread, its point
// coefficients first (read several times), then PrismFx's own.
// Tiles of blockDim elements in two passes, so that a launch shape means the same
// elements per block as in the other plane-major kernels.
template <int KIND, int CPQ, int OUTL>
__global__ void __launch_bounds__(256) __maxnreg__(KIND == POISSON ? 128 : (CPQ ? 168 : 255))
    plane_pair_kernel(const ElemParams p, const __grid_constant__ TmaMaps, const __grid_constant__ CoefFn) {
    extern __shared__ __align__(128) unsigned char smem[];
    double *own = reinterpret_cast<double *>(smem) + (KIND == GENERIC ? threadIdx.x * 60 : 0);
    const double *C = static_cast<const double *>(p.C);
    double *Aout = static_cast<double *>(p.A);
    double *Bout = static_cast<double *>(p.B);
    grid_wait();
    const int sub = threadIdx.x & 1;
    const int64_t ntiles = (p.n + blockDim.x - 1) / blockDim.x;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        if (p.skip_mod > 0 && tile % p.skip_mod == 0) {   // injected fault: no load, no store
            if (threadIdx.x == 0) atomicOr(p.status, ST_SKIPPED_TILES);
            continue;
        }
        for (int pass = 0; pass < 2; ++pass) {
            const int64_t e = tile * blockDim.x + pass * (blockDim.x / 2) + threadIdx.x / 2;
            const bool active = e < p.n;
            const unsigned mask = __ballot_sync(0xFFFFFFFFu, active);
            if (!active) continue;
            const PlaneSrc<double> xs{p.X + e, p.xs}, cg{C + e, p.cs};
            double A[18], b[3];
            bool poor = false;
            uint8_t fl;
            if constexpr (KIND == GENERIC && CPQ) {
#pragma unroll 20
                for (int j = 0; j < 60; ++j) own[j] = ld_stream(C + (60 * sub + j) * p.cs + e);
                fl = ElemMath<PRISM, KIND, FP64, Q_PRISM6, CPQ>::run_pair(xs, SmemSrc<double>{own - 60 * sub, 1}, xs, cg,
                                                                          own, A, b, poor, sub, mask);
            } else {
                fl = ElemMath<PRISM, KIND, FP64, Q_PRISM6, CPQ>::run_pair(xs, cg, xs, cg, own, A, b, poor, sub, mask);
            }
            if (p.flags && sub == 0) p.flags[e] = fl;
#pragma unroll
            for (int j = 0; j < 18; ++j) {
                const int k0 = pair_entry<KIND, FP64>(j, 0), k1 = pair_entry<KIND, FP64>(j, 1);
                if (!out_packed(OUTL)) {
                    st_stream(Aout + (sub ? k1 : k0) * p.os + e, A[j]);
                } else if (sub ? k1 / 6 <= k1 % 6 : k0 / 6 <= k0 % 6) {
                    st_stream(Aout + (sub ? packed_index(6, k1 / 6, k1 % 6) : packed_index(6, k0 / 6, k0 % 6)) * p.os + e,
                              A[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) st_stream(Bout + (3 * sub + j) * p.os + e, b[j]);
        }
    }
}

}  // namespace fe

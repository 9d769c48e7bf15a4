// FP64 tetrahedra in element-contiguous order, one warp at a time: each warp
// takes 32 consecutive elements from staged records to stored results on its own,
// with no block barrier, and its next records travel while it computes.
#pragma once
#include "fe_kernels.cuh"

namespace fe {

// Four doubles to dst: one 32-byte store (a whole sector) when dst allows.
__device__ __forceinline__ void st_row4(double *dst, const double v[4], bool vec32) {
    if (vec32) {
        asm volatile("st.global.cs.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(dst), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3])
                     : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) __stcs(dst + i, v[i]);
    }
}

// An element's record in shared memory on a 16-byte boundary, NR values: read in
// pairs where four consecutive values are taken (a multiple of 4 first).
template <int NR> struct RecSrc {
    const double *base;
    __device__ __forceinline__ double operator()(int j) const { return base[j]; }
};
template <int NR> __device__ __forceinline__ void fx_quad(const RecSrc<NR> &s, int j, double v[4]) {
    static_assert(NR % 4 == 0, "whole pairs");
    const double2 a = *reinterpret_cast<const double2 *>(s.base + j);
    const double2 b = *reinterpret_cast<const double2 *>(s.base + j + 2);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
    v[3] = b.y;
}

// One element outside the fixed-point windows, on the double pipe from global
// memory (its staged record may be gone).
template <int KIND, int QUAD, int CPQ> __device__ __forceinline__ void stream_double_elem(const ElemParams &p, int64_t e) {
    constexpr int NC = ElemCfg<TET, KIND, FP64, QUAD, CPQ>::NC;
    using EM = ElemMath<TET, KIND, FP64, QUAD, CPQ>;
    double A[16], b[4];
    const uint8_t fl = EM::run_double(Src<AOS, double>{p.X + e * 12, 0},
                                      Src<AOS, double>{static_cast<const double *>(p.C) + e * NC, 0}, A, b);
    double *Ao = static_cast<double *>(p.A) + e * 16, *Bo = static_cast<double *>(p.B) + e * 4;
#pragma unroll
    for (int k = 0; k < 16; ++k) Ao[k] = A[k];
#pragma unroll
    for (int k = 0; k < 4; ++k) Bo[k] = b[k];
    if (p.flags) p.flags[e] = fl;
}

// Bound by the double pipe (the edge differences and one conversion per result, 5
// issue slots and 64 pipe cycles per warp each) and by instruction issue; a tile
// kernel that stages, computes, synchronises and stores in turn left the warps
// waiting on copies and barriers for a fifth of the time and held all 20 results
// in registers until the tile's inputs were read. Here:
//  - a warp's records (96 + 8 NC bytes per element) come by bulk copies on the
//    warp's own barrier; the copies of its next 32 elements are issued as soon as
//    the coefficients are consumed (TetFx::columns), half way through an element;
//  - rows of A^e leave as they are formed, one 32-byte store per row and lane;
//    every 32-byte sector is written whole.
// skip_mod and the tile order are those of elem_tiles: tiles of blockDim elements.
template <int KIND, int QUAD, int CPQ> __device__ __forceinline__ void stream_tiles(const ElemParams &p) {
    constexpr int NC = ElemCfg<TET, KIND, FP64, QUAD, CPQ>::NC;
    using EM = ElemMath<TET, KIND, FP64, QUAD, CPQ>;
    constexpr bool MASS2 = QUAD == Q_TET4;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint64_t bars[16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t *bar = &bars[warp];
    if (lane == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    __syncwarp();
    grid_wait();
    double *sX = reinterpret_cast<double *>(smem) + warp * 32 * (12 + NC);
    double *sC = sX + 32 * 12;
    const double *C = static_cast<const double *>(p.C);
    double *Aout = static_cast<double *>(p.A), *Bout = static_cast<double *>(p.B);
    const bool x16 = aligned16(p.X, 0), c16 = aligned16(C, 0);
    const bool o32 = ((reinterpret_cast<uintptr_t>(Aout) | reinterpret_cast<uintptr_t>(Bout)) & 31u) == 0;
    const int64_t B = blockDim.x, ntiles = (p.n + B - 1) / B;

    // the next tile at or after `tile` of this block (past ntiles: none)
    auto next_tile = [&](int64_t tile) {
        while (p.skip_mod > 0 && tile < ntiles && tile % p.skip_mod == 0) {   // injected fault: no load, no store
            if (threadIdx.x == 0) atomicOr(p.status, ST_SKIPPED_TILES);
            tile += gridDim.x;
        }
        return tile;
    };
    // stage this warp's records of a tile; true if a bulk copy was issued
    auto stage = [&](int64_t tile) -> bool {
        const int64_t e0 = tile * B + warp * 32;
        const int64_t left = p.n - e0;
        if (tile >= ntiles || left <= 0) return false;
        const int nb = left < 32 ? int(left) : 32;
        const bool tC = c16 && (nb * NC) % 2 == 0;   // whole 16-byte units (12 coordinates always are)
        if ((x16 || tC) && lane == 0) {
            fence_proxy_async_smem();
            mbar_expect_tx(bar, (x16 ? nb * 96u : 0u) + (tC ? nb * NC * 8u : 0u));
            if (x16) bulk_g2s(sX, p.X + e0 * 12, nb * 96u, bar);
            if (tC) bulk_g2s(sC, C + e0 * NC, nb * NC * 8u, bar);
        }
        if (!x16)
            for (int i = lane; i < nb * 12; i += 32) sX[i] = p.X[e0 * 12 + i];
        if (!tC)
            for (int i = lane; i < nb * NC; i += 32) sC[i] = C[e0 * NC + i];
        return x16 || tC;
    };

    unsigned phase = 0;
    int64_t tile = next_tile(blockIdx.x);
    bool bulk = stage(tile);
    while (tile < ntiles) {
        const int64_t e = tile * B + threadIdx.x;
        const bool active = e < p.n;
        if (bulk) {
            const bool ok = mbar_wait_bounded(bar, phase, p.status);
            phase ^= 1u;
            if (!__all_sync(0xFFFFFFFFu, ok)) {
                // a copy did not land: wait once more (bounded) so nothing is in flight
                mbar_wait_bounded(bar, phase ^ 1u, nullptr);
                return;
            }
        }
        __syncwarp();
        TetFx fx;
        double b[4];
        bool ok = false;
        [[maybe_unused]] TetFx::Rows R;
        if (active) {
            const RecSrc<12> xs{sX + lane * 12};
            const RecSrc<NC> cs{sC + lane * NC};
            ok = fx.geometry(xs);
            if (ok) {
                // (the tests of evenness in one branch: 6M generic 537.6 us, with a branch
                // each 541.8, without them 531)
                if constexpr (KIND == POISSON) {
                    ok = fx.even_rows();
                    EM::poisson_b(fx.volume(), cs, b);
                } else {
                    ok = (fx.even_rows() & fx.even(cs)) && fx.template columns<MASS2>(cs, R, b);
                }
            }
            if (ok) {
                st_row4(Bout + e * 4, b, o32);
                if (p.flags) p.flags[e] = fx.neg ? 2 : 0;
            }
        }
        __syncwarp();   // every record read
        tile = next_tile(tile + gridDim.x);
        bulk = stage(tile);
        if (active) {
            if (ok) {
                double *Ae = Aout + e * 16;
                if constexpr (KIND == POISSON) {
                    double A[16];
                    ok = fx.laplace(A);
#pragma unroll
                    for (int r = 0; r < 4; ++r) st_row4(Ae + 4 * r, A + 4 * r, o32);
                } else {
                    Fx2 fa[3][3];
                    fx.scaled(fa);
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        double A[4];
                        fx.template row<MASS2>(R, fa, r, A);
                        st_row4(Ae + 4 * r, A, o32);
                    }
                }
            }
            if (!ok) stream_double_elem<KIND, QUAD, CPQ>(p, e);   // over what a test after the stores leaves
        }
    }
}

// Registers: generic 128 (3M TET4: 104 registers 10.61, 128 10.85, 144 10.27, 168 9.89
// Gelem/s: above, fewer warps; below, spills and fewer independent chains),
// Laplace 64 (TET1: 48 18.2, 56 19.05, 64 19.1, 80 18.7); before the tests of evenness, which
// take 1% (6M generic 531 -> 538 us, 2M Laplace 105.0 -> 105.7).
template <int KIND, int QUAD, int CPQ>
__global__ void __launch_bounds__(512) __maxnreg__(KIND == POISSON ? 64 : 128)
    stream_kernel_f64t(const ElemParams p, const __grid_constant__ TmaMaps, const __grid_constant__ CoefFn) {
    stream_tiles<KIND, QUAD, CPQ>(p);
}

// FP64 tetrahedra: the warp-at-a-time kernel for element-contiguous records whose
// contractions run in fixed point, else the tile kernel.
template <int KIND, int QUAD, int CPQ, int INL, int OUTL> const void *f64_tet_kernel() {
    if constexpr (INL == AOS && OUTL == AOS && (CPQ == 0 || (CPQ == 1 && KIND == POISSON)))
        return reinterpret_cast<const void *>(&stream_kernel_f64t<KIND, QUAD, CPQ>);
    else if constexpr (INL == SOA && out_soa(OUTL) && plane_mapped(TET, KIND, FP64, CPQ))
        return nullptr;
    else
        return reinterpret_cast<const void *>(&elem_kernel_f64t<KIND, QUAD, CPQ, INL, OUTL>);
}

}  // namespace fe

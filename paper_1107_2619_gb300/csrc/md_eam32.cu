// Mixed-precision EAM passes as stand-alone kernels (md_eam_forces, md_tune); one item
// (lane of an atom) per thread.  The arithmetic is in md_passes.cuh.
#include <cuda_runtime.h>

#include "md_passes.cuh"

namespace mdk {

namespace {

template <int T, int KIND, bool MULTI>
__global__ void __launch_bounds__(kThreads) k_density32(Atoms A, Pot P) {
    if (!eam::begin_density(A.flags)) return;
    ps::density32_item<T, KIND, MULTI>(A, P, A.boxes, (long long)blockIdx.x * kThreads + threadIdx.x);
}

template <int T, int KIND, bool MULTI, bool ENERGY>
__global__ void __launch_bounds__(kThreads) k_force32(Atoms A, Pot P, double half_dt, int kick) {
    if (eam::timed_out(A.flags)) return;
    double part[kPartials];
#pragma unroll
    for (int q = 0; q < kPartials; q++) part[q] = 0.0;
    ps::force32_item<T, KIND, MULTI, ENERGY>(A, P, A.boxes, (long long)blockIdx.x * kThreads + threadIdx.x,
                                             half_dt, kick != 0, part);
    if (ENERGY) eam::block_partials(part, A.partials, A.part_stride);
}

template <int T>
void density_t(const Atoms &A, const Pot &P, cudaStream_t s) {
    const int nb = A.n > 0 ? eam::blocks_for_lanes<T>(A.n) : 1;
    if (P.kind == MD_POT_FS_ANALYTIC) k_density32<T, MD_POT_FS_ANALYTIC, false><<<nb, kThreads, 0, s>>>(A, P);
    else if (P.kind == MD_POT_KNOTS && P.ns == 1) k_density32<T, MD_POT_KNOTS, false><<<nb, kThreads, 0, s>>>(A, P);
    else if (P.kind == MD_POT_KNOTS) k_density32<T, MD_POT_KNOTS, true><<<nb, kThreads, 0, s>>>(A, P);
    else if (P.ns == 1) k_density32<T, MD_POT_TABLES, false><<<nb, kThreads, 0, s>>>(A, P);
    else k_density32<T, MD_POT_TABLES, true><<<nb, kThreads, 0, s>>>(A, P);
}

template <int T, bool ENERGY>
void force_te(const Atoms &A, const Pot &P, double half_dt, int kick, cudaStream_t s) {
    const int nb = eam::blocks_for_lanes<T>(A.n);
    if (P.kind == MD_POT_FS_ANALYTIC)
        k_force32<T, MD_POT_FS_ANALYTIC, false, ENERGY><<<nb, kThreads, 0, s>>>(A, P, half_dt, kick);
    else if (P.kind == MD_POT_KNOTS && P.ns == 1)
        k_force32<T, MD_POT_KNOTS, false, ENERGY><<<nb, kThreads, 0, s>>>(A, P, half_dt, kick);
    else if (P.kind == MD_POT_KNOTS)
        k_force32<T, MD_POT_KNOTS, true, ENERGY><<<nb, kThreads, 0, s>>>(A, P, half_dt, kick);
    else if (P.ns == 1)
        k_force32<T, MD_POT_TABLES, false, ENERGY><<<nb, kThreads, 0, s>>>(A, P, half_dt, kick);
    else
        k_force32<T, MD_POT_TABLES, true, ENERGY><<<nb, kThreads, 0, s>>>(A, P, half_dt, kick);
}

template <int T>
void force_t(const Atoms &A, const Pot &P, bool kick, bool energy, double half_dt, cudaStream_t s) {
    if (energy) force_te<T, true>(A, P, half_dt, kick, s);
    else force_te<T, false>(A, P, half_dt, kick, s);
}

}  // namespace

cudaError_t launch_density32(const Atoms &A, const Pot &P, int lanes, cudaStream_t s) {
    switch (lanes) {
        case 1: density_t<1>(A, P, s); break;
        case 2: density_t<2>(A, P, s); break;
        case 4: density_t<4>(A, P, s); break;
        case 8: density_t<8>(A, P, s); break;
        case 16: density_t<16>(A, P, s); break;
        case 32: density_t<32>(A, P, s); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_force32(const Atoms &A, const Pot &P, int lanes, bool kick, bool energy, double half_dt,
                           cudaStream_t s) {
    if (A.n == 0) return cudaSuccess;
    switch (lanes) {
        case 1: force_t<1>(A, P, kick, energy, half_dt, s); break;
        case 2: force_t<2>(A, P, kick, energy, half_dt, s); break;
        case 4: force_t<4>(A, P, kick, energy, half_dt, s); break;
        case 8: force_t<8>(A, P, kick, energy, half_dt, s); break;
        case 16: force_t<16>(A, P, kick, energy, half_dt, s); break;
        case 32: force_t<32>(A, P, kick, energy, half_dt, s); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace mdk

// Instantiation and dispatch of the 3D step kernel for one precision policy.
#pragma once

#include "pf.h"
#include "pf_internal.h"
#include "pf_kernels3d_pair.cuh"

namespace pf {

template <class P, int TX, int TY, bool MOVING, int MODE, bool EXT, bool UNIT = false>
static bool run3d(int grid, cudaStream_t s, const StepArgs &a, int *occ)
{
    using R = typename P::real;
    auto kern = k_step3d<P, TX, TY, MOVING, MODE, EXT, UNIT>;
    const int dyn = MOVING ? (int)step3d_moving_smem<R, TX, TY>(a.np, a.wv) : 0;
    // the limit is the function's, shared by every simulation and host thread: always
    // the largest size, so that no launch finds it below its own
    constexpr int dyn_max = MOVING ? (int)step3d_moving_smem<R, TX, TY>(PF_MAX_PARTICLES, true) : 0;
    if (dyn && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_max) != cudaSuccess)
        return false;
    if (occ) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, TX * TY, dyn) != cudaSuccess) n = 0;
        *occ = n;
        return true;
    }
    const DomainDev d1 = a.dom1 ? *a.dom1 : DomainDev{};
    if constexpr (MOVING && MODE == MODE_STEP && sizeof(R) == 4) {
        k_phi3d<P, TX, TY, EXT, true><<<dim3(a.ntiles, 8), TX * TY, 0, s>>>(a, d1, 1);
        count_launches(1);
    }
    kern<<<grid, TX * TY, dyn, s>>>(a, d1);
    count_launches(1);
    return true;
}

// the step of the FP32-arithmetic policies without particles: phi of every
// cell, then the two-cells-per-thread update
template <class P, int TX, int TY, bool EXT, bool UNIT, bool SINGLE>
static bool run3d_pair(int grid, cudaStream_t s, const StepArgs &a, int *occ)
{
    auto kern = k_step3d_pair<P, TX, TY, EXT, UNIT, SINGLE>;
    constexpr int smem = step3d_pair_smem<TX, TY>();
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return false;
    if (occ) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, TX * TY, smem) != cudaSuccess) n = 0;
        *occ = n;
        return true;
    }
    // eight pieces of a tile's planes: enough blocks of the light pass to fill
    // the chip also where the tiles alone would not
    const DomainDev d1 = SINGLE ? *a.dom1 : DomainDev{};
    k_phi3d<P, TX, TY, EXT, SINGLE><<<dim3(a.ntiles, 8), TX * TY, 0, s>>>(a, d1, 2);
    kern<<<grid, TX * TY, smem, s>>>(a, d1);
    count_launches(2);
    return true;
}

template <class P, int TX, int TY, bool EXT>
static bool dispatch3d_ext(bool moving, bool unit, int mode, int grid, cudaStream_t s, const StepArgs &a, int *occ)
{
    if (mode == MODE_MACROS)
        return moving ? run3d<P, TX, TY, true, MODE_MACROS, EXT>(grid, s, a, occ)
                      : run3d<P, TX, TY, false, MODE_MACROS, EXT>(grid, s, a, occ);
    if constexpr (sizeof(typename P::real) == 4) {
        if (!moving && a.dom1)
            return unit ? run3d_pair<P, TX, TY, EXT, true, true>(grid, s, a, occ)
                        : run3d_pair<P, TX, TY, EXT, false, true>(grid, s, a, occ);
        if (!moving)
            return unit ? run3d_pair<P, TX, TY, EXT, true, false>(grid, s, a, occ)
                        : run3d_pair<P, TX, TY, EXT, false, false>(grid, s, a, occ);
    }
    if (moving)
        return unit ? run3d<P, TX, TY, true, MODE_STEP, EXT, true>(grid, s, a, occ)
                    : run3d<P, TX, TY, true, MODE_STEP, EXT>(grid, s, a, occ);
    if constexpr (sizeof(typename P::real) == 8)
        return unit ? run3d<P, TX, TY, false, MODE_STEP, EXT, true>(grid, s, a, occ)
                    : run3d<P, TX, TY, false, MODE_STEP, EXT>(grid, s, a, occ);
    return false;
}

// mode may carry MODE_EXT: a domain of the launch has walls
template <class P, int TX, int TY>
static bool dispatch3d(int tx, int ty, bool moving, int mode, int grid, cudaStream_t s,
                       const StepArgs &a, int *occ)
{
    if (tx != TX || ty != TY) return false;
    const bool ext = (mode & MODE_EXT) != 0, unit = (mode & MODE_UNIT) != 0;
    mode &= ~(MODE_EXT | MODE_CAC | MODE_UNIT);
    return ext ? dispatch3d_ext<P, TX, TY, true>(moving, unit, mode, grid, s, a, occ)
               : dispatch3d_ext<P, TX, TY, false>(moving, unit, mode, grid, s, a, occ);
}

}  // namespace pf

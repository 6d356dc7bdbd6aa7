// Kernel templates of the staggered D_S and D_S^+ sweeps (Sec. 3, plus a mass
// term) on the internal blocked layout; instantiated once per storage type in
// apply_staggered_<type>.cu.  One thread owns one site and R right-hand
// sides: every link is loaded once per thread and applied to its R spinors
// from registers, and every output element is written once.  Consecutive
// blocks cover the right-hand-side groups of the same sites, so the other
// groups find the links in L2.
#pragma once

#include <type_traits>

#include "dirac_internal.h"

namespace dirac {

// CANON: the output goes to the canonical field a.canon (warp_store, whole warps)
template <typename T, int R, bool DAG, bool CANON>
__global__ void __launch_bounds__(256) k_staggered(ApplyArgs a, int ngroups)
{
    const long b = blockIdx.x;
    const int group = (int)(b % ngroups);
    const long p = (b / ngroups) * blockDim.x + threadIdx.x;
    if constexpr (CANON) {
        extern __shared__ __align__(16) unsigned char sm[];
        if (p - (threadIdx.x & 31) >= a.nsites) return;   // a whole warp
        const OutTo to{sm + (threadIdx.x >> 5) * staggered_store_bytes<T, R>(), (int)(threadIdx.x & 31), p < a.nsites};
        staggered_site<T, R, DAG, 0, 0, true>(a, slab_site(a, min(p, a.nsites - 1)), group, to);
    } else {
        if (p >= a.nsites) return;
        staggered_site<T, R, DAG>(a, slab_site(a, p), group);
    }
}

// V_GROUPS: blockDim = (sites, groups); block b covers a run of sites and a
// chunk of gy right-hand-side groups
// LF: link format (0 nine entries per link, 1 two rows, reconstructed)
template <typename T, int R, bool DAG, int MODE, int LF, bool CANON>
__global__ void __launch_bounds__(192, 2) k_staggered_groups(ApplyArgs a, int ngroups, int gy)
{
    const int nchunks = (ngroups + gy - 1) / gy;
    const long b = blockIdx.x;
    const int group = (int)(b % nchunks) * gy + threadIdx.y;
    const long p = (b / nchunks) * blockDim.x + threadIdx.x;
    if constexpr (CANON) {
        extern __shared__ __align__(16) unsigned char sm[];
        if (p - (threadIdx.x & 31) >= a.nsites || group >= ngroups) return;   // a whole warp
        const OutTo to{sm + ((threadIdx.y * blockDim.x + threadIdx.x) >> 5) * staggered_store_bytes<T, R>(),
                       (int)(threadIdx.x & 31), p < a.nsites};
        staggered_site<T, R, DAG, MODE, LF, true>(a, slab_site(a, min(p, a.nsites - 1)), group, to);
    } else {
        if (p >= a.nsites || group >= ngroups) return;
        staggered_site<T, R, DAG, MODE, LF>(a, slab_site(a, p), group);
    }
}

// V_XLAST: V_GROUPS with the x hops last, by lane exchange (staggered_site_xlast);
// the host checked that every warp holds whole x-rows
template <typename T, int R, bool DAG, int MODE, int LF, bool CANON>
__global__ void __launch_bounds__(192, 2) k_staggered_xlast(ApplyArgs a, int ngroups, int gy)
{
    const int nchunks = (ngroups + gy - 1) / gy;
    const long b = blockIdx.x;
    const int group = (int)(b % nchunks) * gy + threadIdx.y;
    const long p = (b / nchunks) * blockDim.x + threadIdx.x;
    if (p >= a.nsites || group >= ngroups) return;   // whole warps
    if constexpr (CANON) {
        extern __shared__ __align__(16) unsigned char sm[];
        const OutTo to{sm + ((threadIdx.y * blockDim.x + threadIdx.x) >> 5) * staggered_store_bytes<T, R>(),
                       (int)(threadIdx.x & 31), true};
        staggered_site_xlast<T, R, DAG, MODE, LF, true>(a, slab_site(a, p), threadIdx.x & 31, group, to);
    } else {
        staggered_site_xlast<T, R, DAG, MODE, LF>(a, slab_site(a, p), threadIdx.x & 31, group);
    }
}

template <typename T, int R>
cudaError_t staggered_go(bool dag, const ApplyArgs& a, LaunchCfg c, cudaStream_t st)
{
    const int block = c.block;
    const int ngroups = (a.Nv + R - 1) / R;
    if constexpr (sizeof(T) != 8) {
    if (c.variant == V_XLAST) {
        const int gy = groups_per_block(block, ngroups);
        const long nb = ((a.nsites + block - 1) / block) * (long)((ngroups + gy - 1) / gy);
        const bool dv = a.diag_vf != nullptr;
        const int mode = (a.Nv % R != 0 || (a.diag_v != nullptr && !dv)) ? 0 : (dv ? 2 : 1);
        auto launch_lf = [&](auto m, auto lf) {
            constexpr int M = decltype(m)::value;
            constexpr int LF = decltype(lf)::value;
            if constexpr (sizeof(T) >= 4 && M < 2) {
                if (a.canon) {
                    const size_t sm = (size_t)(block / 32 * gy) * staggered_store_bytes<T, R>();
                    if (dag) k_staggered_xlast<T, R, true, M, LF, true><<<(unsigned)nb, dim3(block, gy), sm, st>>>(a, ngroups, gy);
                    else k_staggered_xlast<T, R, false, M, LF, true><<<(unsigned)nb, dim3(block, gy), sm, st>>>(a, ngroups, gy);
                    return;
                }
            }
            if (dag) k_staggered_xlast<T, R, true, M, LF, false><<<(unsigned)nb, dim3(block, gy), 0, st>>>(a, ngroups, gy);
            else k_staggered_xlast<T, R, false, M, LF, false><<<(unsigned)nb, dim3(block, gy), 0, st>>>(a, ngroups, gy);
        };
        auto launch = [&](auto m) {
            if (c.fmt == 1) launch_lf(m, std::integral_constant<int, 1>{});
            else launch_lf(m, std::integral_constant<int, 0>{});
        };
        if (mode == 1) launch(std::integral_constant<int, 1>{});
        else if (mode == 2) launch(std::integral_constant<int, 2>{});
        else launch(std::integral_constant<int, 0>{});
        return cudaGetLastError();
    }
    }
    if (c.variant == V_GROUPS) {
        const int gy = groups_per_block(block, ngroups);
        const long nb = ((a.nsites + block - 1) / block) * (long)((ngroups + gy - 1) / gy);
        const bool dv = sizeof(T) == 8 ? a.diag_v != nullptr : a.diag_vf != nullptr;
        const int mode = (a.Nv % R != 0 || (a.diag_v != nullptr && !dv)) ? 0 : (dv ? 2 : 1);
        auto launch_lf = [&](auto m, auto lf) {
            constexpr int M = decltype(m)::value;
            constexpr int LF = decltype(lf)::value;
            if constexpr (sizeof(T) >= 4 && M < 2) {
                if (a.canon) {
                    const size_t sm = (size_t)(block / 32 * gy) * staggered_store_bytes<T, R>();
                    if (dag) k_staggered_groups<T, R, true, M, LF, true><<<(unsigned)nb, dim3(block, gy), sm, st>>>(a, ngroups, gy);
                    else k_staggered_groups<T, R, false, M, LF, true><<<(unsigned)nb, dim3(block, gy), sm, st>>>(a, ngroups, gy);
                    return;
                }
            }
            if (dag) k_staggered_groups<T, R, true, M, LF, false><<<(unsigned)nb, dim3(block, gy), 0, st>>>(a, ngroups, gy);
            else k_staggered_groups<T, R, false, M, LF, false><<<(unsigned)nb, dim3(block, gy), 0, st>>>(a, ngroups, gy);
        };
        auto launch = [&](auto m) {
            // two-row links are built for FP32 and 16-bit storage only
            if constexpr (sizeof(T) != 8) {
                if (c.fmt == 1) return launch_lf(m, std::integral_constant<int, 1>{});
            }
            launch_lf(m, std::integral_constant<int, 0>{});
        };
        if (mode == 1) launch(std::integral_constant<int, 1>{});
        else if (mode == 2) launch(std::integral_constant<int, 2>{});
        else launch(std::integral_constant<int, 0>{});
        return cudaGetLastError();
    }
    const long nblk = ((a.nsites + block - 1) / block) * (long)ngroups;
    if constexpr (sizeof(T) >= 4 && (R < 6 || sizeof(T) == 4)) {
        if (a.canon) {
            const size_t sm = (size_t)(block / 32) * staggered_store_bytes<T, R>();
            if (dag) k_staggered<T, R, true, true><<<(unsigned)nblk, block, sm, st>>>(a, ngroups);
            else k_staggered<T, R, false, true><<<(unsigned)nblk, block, sm, st>>>(a, ngroups);
            return cudaGetLastError();
        }
    }
    if (dag) k_staggered<T, R, true, false><<<(unsigned)nblk, block, 0, st>>>(a, ngroups);
    else k_staggered<T, R, false, false><<<(unsigned)nblk, block, 0, st>>>(a, ngroups);
    return cudaGetLastError();
}

template <typename T>
cudaError_t staggered_go_T(bool dag, const ApplyArgs& a, LaunchCfg c, cudaStream_t st)
{
    if (c.variant != V_DIRECT && c.variant != V_GROUPS && c.variant != V_XLAST) return cudaErrorInvalidValue;
    switch (c.R) {
    case 1: return staggered_go<T, 1>(dag, a, c, st);
    case 2: return staggered_go<T, 2>(dag, a, c, st);
    case 6: return staggered_go<T, 6>(dag, a, c, st);
    case 4: return staggered_go<T, 4>(dag, a, c, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace dirac

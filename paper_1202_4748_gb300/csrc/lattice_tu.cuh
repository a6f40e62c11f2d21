// Shared body of the per-lattice translation units: tile-shape table and the
// launchers for the step, init, gather/scatter and observable-site kernels.
#pragma once

#include <type_traits>

#include "lattice_kernels.cuh"
#include "lb_launch.h"
#include "step_kernel_modeq3.cuh"
#include "step_kernel_pair.cuh"
#include "step_kernel_split.cuh"
#include "step_kernel_strip_pair.cuh"
#include "step_kernels.cuh"

namespace lbf {

template <class Real>
StepArgs<Real> step_args(const StepLaunch& a) {
    StepArgs<Real> A;
    A.sys = a.sys;
    A.phys = static_cast<const SysPhys<Real>*>(a.phys);
    A.tiles = a.tiles;
    A.fin = static_cast<const Real*>(a.fin);
    A.fout = static_cast<Real*>(a.fout);
    A.step_ptr = a.step_ptr;
    A.k = a.k;
    A.status = a.status;
    A.zc = a.zc;
    A.early = a.early;
    return A;
}

template <class L, int CP, class Real, int TX, int TY, int TZ, int MODE>
cudaError_t step_one_mode(const StepLaunch& a, cudaStream_t st) {
    const StepArgs<Real> A = step_args<Real>(a);
    step_kernel<L, CP, Real, TX, TY, TZ, MODE><<<a.n_tiles, TX * TY * TZ, 0, st>>>(A);
    return cudaGetLastError();
}

// Row-marching strips (D2Q9, modified equilibrium): tiles of SW sites x a.zc
// rows, a warp per 32 sites of a tile.  One warp per CTA: everything that is the
// same in the warp's lanes (the system's records, the tile, the noise key) is
// then the same in the CTA and needs no register per lane.  With four warps per
// CTA the two-site kernel took 168 registers, now 92: 20 warps per SM instead
// of 12.
template <class L, int CP, class Real, int MINB, int MODE, int SW>
cudaError_t step_strip_mode(const StepLaunch& a, cudaStream_t st) {
    step_kernel_strip<L, CP, Real, MINB, MODE, SW><<<a.n_tiles * (SW / 32), 32, 0, st>>>(step_args<Real>(a));
    return cudaGetLastError();
}
template <class L, int CP, class Real, int MINB, int SW = 32>
cudaError_t step_strip(const StepLaunch& a, cudaStream_t st) {
    constexpr int MB = sizeof(Real) == 4 && MINB > 0 ? MINB : 1;   // FP64 keeps its registers
    if (a.bgk_only == 2) return step_strip_mode<L, CP, Real, MB, 2, SW>(a, st);
    if (a.bgk_only == 1) return step_strip_mode<L, CP, Real, MB, 1, SW>(a, st);
    return step_strip_mode<L, CP, Real, MB, 0, SW>(a, st);
}

// Two-site strips (D2Q9, modified equilibrium, FP32, every mode at tau = 1,
// every x side a multiple of 4) on tiles of 64 sites x a.zc rows; any other run
// of the same tiles takes the one-site strips, two warps per tile.
template <class L, int CP, class Real, int MINB>
cudaError_t step_strip2(const StepLaunch& a, cudaStream_t st) {
    if constexpr (sizeof(Real) == 4 && CP == MODEQ) {
        if (a.bgk_only == 2 && a.pair_ok) {
            step_kernel_strip_pair<MINB><<<a.n_tiles, 32, 0, st>>>(step_args<float>(a));
            return cudaGetLastError();
        }
    }
    return step_strip<L, CP, Real, MINB, 64>(a, st);
}

// z-marching launches (FP32, every mode at tau = 1): columns of TX x TY sites,
// chunks of a.zc planes, a register budget for MINB resident CTAs per SM; the
// Guo form, and the modified equilibrium on its radius-1 footprint.
template <class L, int TX, int TY, int MINB>
cudaError_t step_z(const StepLaunch& a, cudaStream_t st) {
    step_kernel_z<L, TX, TY, MINB><<<a.n_tiles, TX * TY, 0, st>>>(step_args<float>(a));
    return cudaGetLastError();
}
template <class L, int TX, int TY, int MINB>
cudaError_t step_zm(const StepLaunch& a, cudaStream_t st) {
    constexpr int MB = MINB < 2 ? 2 : MINB;
    step_kernel_zm<L, TX, TY, MB><<<a.n_tiles, TX * TY, 0, st>>>(step_args<float>(a));
    return cudaGetLastError();
}

// Warp-specialised launch (fully relaxed Guo path, FP32): TX x TY consumer
// threads and PW producer warps per CTA; STG = 1 stages the footprint with
// bulk copies (a dynamic shared-memory stage), 0 with plain loads.
template <class L, int TX, int TY, int PW, int MINB, int STG>
cudaError_t step_ws(const StepLaunch& a, cudaStream_t st) {
    const StepArgs<float> A = step_args<float>(a);
    size_t dyn = 0;
    if constexpr (STG == 1) {
        dyn = BulkStage<L, TX, TY, PW>::bytes;
        static PerDevice attr;                 // once per instantiation and device
        cudaError_t e = cudaSuccess;
        const int set = attr.get(current_device(), [&] {
            auto k = step_kernel_ws<L, TX, TY, PW, MINB, STG>;
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(dyn));
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         int(cudaSharedmemCarveoutMaxShared));
            return e == cudaSuccess ? 1 : 0;
        });
        if (!set) return e;
    }
    step_kernel_ws<L, TX, TY, PW, MINB, STG><<<a.n_tiles, TX * TY + 32 * PW, dyn, st>>>(A);
    return cudaGetLastError();
}

// Paired-site warp-specialised launch (fully relaxed path on D3Q19, FP32,
// every nx a multiple of 4; the Guo form, or CP = MODEQ the modified
// equilibrium): TX TY / 2 consumer threads and PW producer warps
// per CTA, rings of R planes (and, STG = 3, the producers' staging area) in
// dynamic shared memory.
template <int TX, int TY, int PW, int MINB, int R, int STG, int CP = GUO>
cudaError_t step_pair(const StepLaunch& a, cudaStream_t st) {
    const StepArgs<float> A = step_args<float>(a);
    constexpr size_t dyn = PairSmem<TX, TY, PW, R, STG, CP>::bytes;
    static PerDevice usable;                   // once per instantiation and device: 1 usable, -1 not
    cudaError_t e = cudaSuccess;
    const int state = usable.get(current_device(), [&] {
        auto k = step_kernel_pair<TX, TY, PW, MINB, R, STG, CP>;
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, k);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(dyn));
        // (no carve-out preference: the rings need a fraction of the SM's
        // shared memory, and the producers' load misses are staged in L1)
        if (e != cudaSuccess) return 0;
        // the register split must balance against the launch count it assumes
        return !PairRegs<TX, TY, PW, MINB, STG>::split || fa.numRegs == PairRegs<TX, TY, PW, MINB, STG>::launch ? 1 : -1;
    });
    if (!state) return e;
    if (state < 0) {
        if constexpr (CP == MODEQ) return step_zm<D3Q19, TX, TY, MINB>(a, st);
        else return step_ws<D3Q19, TX, TY, PW, 1, 0>(a, st);
    }
    step_kernel_pair<TX, TY, PW, MINB, R, STG, CP><<<a.n_tiles, TX * TY / 2 + 32 * PW, dyn, st>>>(A);
    return cudaGetLastError();
}

// Launch with programmatic stream serialisation: the kernel may start before
// its predecessor on the stream has ended and orders itself with grid_wait.
template <class... P, class... A>
cudaError_t launch_dependent(void (*kernel)(P...), unsigned grid, unsigned block, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = st;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Moment pass of the split step: quads of sites where every nx is a multiple of
// 4 (FP32), else single sites; small CTAs when the items are small (few of them).
template <class L, class Real, bool J>
cudaError_t step_moments(const StepLaunch& a, cudaStream_t st) {
    const Real* f = static_cast<const Real*>(a.fin);
    Real* mom = static_cast<Real*>(a.mom);
    if constexpr (sizeof(Real) == 4) {
        if (a.pair_ok) {
            if (a.small_items)
                return launch_dependent(moments_quad_kernel<L, J, 64>, a.n_site_items, 64, st, a.sys, a.site_items, f,
                                        mom, a.n_sites, a.early);
            return launch_dependent(moments_quad_kernel<L, J, 256>, a.n_site_items, 256, st, a.sys, a.site_items, f,
                                    mom, a.n_sites, a.early);
        }
    }
    return launch_dependent(moments_kernel<L, Real, J, 256>, a.n_site_items, 256, st, a.sys, a.site_items, f, mom,
                            a.n_sites, a.early);
}

// Split step on D3Q19: the moment pass over the site items, then the collision
// of 16 x 8 columns (FP64: 8 x 8 where they leave fewer lanes outside the
// systems) in chunks of a.zc planes.  4 resident CTAs, 128 registers: no spills
// fully relaxed; other rates, which keep the populations to the end, spill 12 to 60
// bytes, and FP32 with a rate per mode takes 4 x 64^3 in 63.5 us (3 CTAs, 168
// registers, no spills: 67.3), 160^3 in 229 (233).  Fully relaxed, 5 CTAs spill 8
// bytes and give 134.5 us for 136.5 on 2.6 M odd-sided sites but 198 for 192 on
// 4 x 99^3; FP64 hides its latencies better with 4 than with 2 (64^3 190 -> 173 us).
template <int MODE, int CP, class Real, int TX>
cudaError_t step_split_columns(const StepLaunch& a, cudaStream_t st) {
    using V = typename std::conditional<std::is_same<Real, float>::value, float2, double>::type;
    constexpr int MINB = 4 * (16 / TX);
    const cudaError_t e = step_moments<D3Q19, Real, MODE == 2 && sizeof(Real) == 4>(a, st);
    if (e != cudaSuccess) return e;
    return launch_dependent(collide_march_kernel<MODE, CP, V, TX, 8, MINB>, a.n_tiles, 8 * TX, st,
                            step_args<Real>(a), static_cast<const Real*>(a.mom), a.n_sites);
}
template <int MODE, int CP, class Real>
cudaError_t step_split_mode(const StepLaunch& a, cudaStream_t st) {
    if constexpr (sizeof(Real) == 8) {
        if (a.narrow) return step_split_columns<MODE, CP, Real, 8>(a, st);
    }
    return step_split_columns<MODE, CP, Real, 16>(a, st);
}
template <int CP, class Real>
cudaError_t step_split(const StepLaunch& a, cudaStream_t st) {
    if (a.bgk_only == 2) return step_split_mode<2, CP, Real>(a, st);
    if (a.bgk_only == 1) return step_split_mode<1, CP, Real>(a, st);
    return step_split_mode<0, CP, Real>(a, st);
}

template <class L, int CP, class Real, int TX, int TY, int TZ>
cudaError_t step_one(const StepLaunch& a, cudaStream_t st) {
    if (a.bgk_only == 2) return step_one_mode<L, CP, Real, TX, TY, TZ, 2>(a, st);
    if (a.bgk_only == 1) return step_one_mode<L, CP, Real, TX, TY, TZ, 1>(a, st);
    return step_one_mode<L, CP, Real, TX, TY, TZ, 0>(a, st);
}

template <class L, class Real>
cudaError_t init_feq_any(int coupling, const SysDev* sys, const int4* items, int n_items, const double* d,
                         const double* dbar, void* fbuf, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    if (coupling == MODEQ) {
        init_feq_kernel<L, MODEQ, Real><<<n_items, AUX_THREADS, 0, st>>>(sys, items, d, dbar, static_cast<Real*>(fbuf));
    } else {
        init_feq_kernel<L, GUO, Real><<<n_items, AUX_THREADS, 0, st>>>(sys, items, d, dbar, static_cast<Real*>(fbuf));
    }
    return cudaGetLastError();
}

template <class L, class Real>
cudaError_t gather_any(const SysDev* sys, int s, int i0, int ni, int64_t n, const void* fbuf, double* out, cudaStream_t st) {
    const dim3 grid(unsigned((n + AUX_THREADS - 1) / AUX_THREADS), unsigned(ni));
    gather_kernel<L, Real><<<grid, AUX_THREADS, 0, st>>>(sys, s, i0, static_cast<const Real*>(fbuf), out);
    return cudaGetLastError();
}

template <class L, class Real>
cudaError_t scatter_any(const SysDev* sys, int s, int i0, int ni, int64_t n, const double* in, void* fbuf, cudaStream_t st) {
    const dim3 grid(unsigned((n + AUX_THREADS - 1) / AUX_THREADS), unsigned(ni));
    scatter_kernel<L, Real><<<grid, AUX_THREADS, 0, st>>>(sys, s, i0, in, static_cast<Real*>(fbuf));
    return cudaGetLastError();
}

template <class L, class Real>
cudaError_t obs_site_any(const SysDev* sys, const int4* items, int n_items, const void* fbuf, double* d,
                         double* partial, double* jout, int64_t jstride, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    obs_site_kernel<L, Real><<<n_items, AUX_THREADS, 0, st>>>(sys, items, static_cast<const Real*>(fbuf), d, partial,
                                                              jout, jstride);
    return cudaGetLastError();
}

}  // namespace lbf

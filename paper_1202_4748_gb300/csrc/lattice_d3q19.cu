// D3Q19 instantiations (3-D variant): the Guo-forced form with the Landau
// pressure in the equilibrium and the modified equilibrium carried to three
// dimensions, FP64 and FP32-deviation storage.
#include <utility>

#include "lattice_tu.cuh"

namespace lbf {

namespace {
// (x, y, z-chunk, resident CTAs per SM, producer warps, staging, sites per
// consumer thread) of the z-marching kernels of the fully relaxed FP32 path:
// producer warps 0 = every thread stages and collides its own column; > 0 =
// warp-specialised kernel, whose producers stage the footprint with plain
// loads (staging 0) or with bulk copies into shared memory (staging 1; systems
// that do not allow it run the staging-0 kernel of the same tile); the paired
// kernel stages aligned quads in registers (0) or with cp.async in shared
// memory (3).  Two sites per consumer thread: the paired kernel (x-adjacent
// site pairs, paired FP32 arithmetic; ensembles with an nx that is not a
// multiple of 4 run the one-site warp-specialised kernel of the same tile).
// The 16 x 8 rows with 4 resident CTAs are the split step (a moment pass, then
// collision columns, two sites stacked in z per thread), which FP64 runs and
// other relaxation rates take whatever the row, with the row's z-chunk.  The
// first entry is the default.
constexpr int kTiles[][kVariantCols] = {
    {32, 8, 32, 3, 4, 3, 2}, {32, 8, 64, 3, 4, 3, 2}, {16, 16, 32, 3, 4, 3, 2}, {16, 16, 64, 3, 4, 3, 2},
    {32, 8, 32, 2, 4, 0, 2}, {16, 16, 32, 2, 4, 0, 2},
    {32, 8, 64, 2, 4, 0, 2}, {16, 8, 32, 3, 4, 0, 1},  {16, 8, 64, 3, 4, 0, 1},  {16, 8, 16, 3, 4, 0, 1},
    {16, 8, 32, 3, 4, 1, 1}, {16, 8, 16, 6, 0, 0, 1},  {16, 8, 32, 6, 0, 0, 1},  {16, 16, 16, 4, 0, 0, 1},
    {16, 16, 32, 4, 0, 0, 1},
    {32, 8, 16, 3, 4, 3, 2}, {32, 8, 8, 3, 4, 3, 2},
    {16, 8, 2, 4, 0, 0, 1},  {16, 8, 4, 4, 0, 0, 1},   {16, 8, 8, 4, 0, 0, 1},   {16, 8, 16, 4, 0, 0, 1},
    {16, 8, 32, 4, 0, 0, 1}};
constexpr int kNumTiles = int(sizeof(kTiles) / sizeof(kTiles[0]));
// ring planes of the paired kernel: 8 with register staging (2 CTAs per SM),
// 4 with cp.async staging (the staging areas share the shared memory)
constexpr int pair_ring(int stg) { return stg == 3 ? 4 : 8; }

// FP32, every mode at tau = 1.
template <int CP, int I>
cudaError_t step_variant(const StepLaunch& a, cudaStream_t st) {
    constexpr int TX = kTiles[I][0], TY = kTiles[I][1], OCC = kTiles[I][3], PW = kTiles[I][4], STG = kTiles[I][5];
    constexpr bool paired = PW > 0 && kTiles[I][6] == 2;
    if constexpr (split_row(kTiles[I])) {
        return cudaErrorInvalidValue;        // the plan runs these rows as the split step
    } else if constexpr (CP == MODEQ) {
        // the modified equilibrium: the paired kernel on the paired cp.async rows (every
        // nx a multiple of 4), else the radius-1 z-marching kernel of the same tile
        if constexpr (paired && STG == 3) {
            if (a.pair_ok) return step_pair<TX, TY, PW, OCC, pair_ring(STG), STG, MODEQ>(a, st);
        }
        return step_zm<D3Q19, TX, TY, OCC>(a, st);
    } else if constexpr (paired) {
        if (a.pair_ok) return step_pair<TX, TY, PW, OCC, pair_ring(STG), STG>(a, st);
        return step_ws<D3Q19, TX, TY, PW, 1, 0>(a, st);
    } else if constexpr (PW > 0) {
        if constexpr (STG == 1) {
            if (a.bulk_ok) return step_ws<D3Q19, TX, TY, PW, OCC, 1>(a, st);
        }
        return step_ws<D3Q19, TX, TY, PW, OCC, 0>(a, st);
    } else {
        return step_z<D3Q19, TX, TY, OCC>(a, st);
    }
}

template <int CP, int... I>
cudaError_t step_tile_of(const StepLaunch& a, cudaStream_t st, std::integer_sequence<int, I...>) {
    using Fn = cudaError_t (*)(const StepLaunch&, cudaStream_t);
    static constexpr Fn table[] = {&step_variant<CP, I>...};
    if (a.tile_id < 0 || a.tile_id >= int(sizeof...(I))) return cudaErrorInvalidValue;
    return table[a.tile_id](a, st);
}

template <int CP>
cudaError_t step_tile(const StepLaunch& a, cudaStream_t st) {
    return step_tile_of<CP>(a, st, std::make_integer_sequence<int, kNumTiles>{});
}
}  // namespace

int tile_shapes_d3q19(int (*out)[kVariantCols], int max) {
    for (int t = 0; t < kNumTiles && t < max; ++t)
        for (int k = 0; k < kVariantCols; ++k) out[t][k] = kTiles[t][k];
    return kNumTiles;
}

cudaError_t launch_step_d3q19(int coupling, int fp32, const StepLaunch& a, cudaStream_t st) {
    if (a.n_tiles == 0) return cudaSuccess;
    if (a.split) {
        if (coupling == MODEQ) return fp32 ? step_split<MODEQ, float>(a, st) : step_split<MODEQ, double>(a, st);
        return fp32 ? step_split<GUO, float>(a, st) : step_split<GUO, double>(a, st);
    }
    return coupling == MODEQ ? step_tile<MODEQ>(a, st) : step_tile<GUO>(a, st);
}

cudaError_t launch_init_feq_d3q19(int coupling, int fp32, const SysDev* sys, const int4* items, int n_items,
                                 const double* d, const double* dbar, void* fbuf, cudaStream_t st) {
    return fp32 ? init_feq_any<D3Q19, float>(coupling, sys, items, n_items, d, dbar, fbuf, st)
                : init_feq_any<D3Q19, double>(coupling, sys, items, n_items, d, dbar, fbuf, st);
}
cudaError_t launch_gather_d3q19(int fp32, const SysDev* sys, int s, int i0, int ni, int64_t n, const void* fbuf, double* out,
                               cudaStream_t st) {
    return fp32 ? gather_any<D3Q19, float>(sys, s, i0, ni, n, fbuf, out, st)
                : gather_any<D3Q19, double>(sys, s, i0, ni, n, fbuf, out, st);
}
cudaError_t launch_scatter_d3q19(int fp32, const SysDev* sys, int s, int i0, int ni, int64_t n, const double* in, void* fbuf,
                                cudaStream_t st) {
    return fp32 ? scatter_any<D3Q19, float>(sys, s, i0, ni, n, in, fbuf, st)
                : scatter_any<D3Q19, double>(sys, s, i0, ni, n, in, fbuf, st);
}
cudaError_t launch_obs_site_d3q19(int fp32, const SysDev* sys, const int4* items, int n_items, const void* fbuf,
                                 double* d, double* partial, double* jout, int64_t jstride, cudaStream_t st) {
    return fp32 ? obs_site_any<D3Q19, float>(sys, items, n_items, fbuf, d, partial, jout, jstride, st)
                : obs_site_any<D3Q19, double>(sys, items, n_items, fbuf, d, partial, jout, jstride, st);
}

}  // namespace lbf

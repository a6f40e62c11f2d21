// Internal host-side interface between the C ABI (api.cu) and the kernel
// translation units.  Plain structs and pointers only.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "lb_device.cuh"
#include "per_device.h"

namespace lbf {

constexpr int AUX_THREADS = 256;        // threads of the auxiliary (non-step) kernels
constexpr int SITES_PER_THREAD = 4;     // sites per thread in a site-pass item

// The calling thread's device (-1: none).
inline int current_device() {
    int d = -1;
    return cudaGetDevice(&d) == cudaSuccess ? d : -1;
}

struct StepLaunch {
    const SysDev* sys;
    const void* phys;       // SysPhys<float> or SysPhys<double> per system
    const int4* tiles;
    int n_tiles;
    const void* fin;
    void* fout;
    const int64_t* step_ptr;
    int k;
    int* status;
    int tile_id;            // index into the lattice's tile-shape table
    int zc;                 // planes per chunk of the z-marching kernels, rows per strip on D2Q9
    int split;              // D3Q19: run the split step
    int narrow;             // in 8 x 8 columns (FP64)
    int early;              // both kernels' CTAs fit on an SM each: each lets the next start at once
    void* mom;              // split step: density and momentum fields, one per n_sites values
    int64_t n_sites;        // sites of the ensemble
    const int4* site_items; // split step: the moment pass's work list
    int n_site_items;
    int small_items;        // the items hold AUX_THREADS sites (else SITES_PER_THREAD times as many)
    int bgk_only;           // 0: per-mode rates; 1: one rate per system; 2: one rate, equal to 1
    int bulk_ok;            // every system allows bulk-copy staging (nx % 4 == 0, nx >= 8, sides >= 3)
    int pair_ok;            // every system has nx % 4 == 0 (the paired-site kernel can run)
};

// Step-kernel variants compiled for each lattice: (x, y, z, resident CTAs per
// SM, producer warps, staging: 0 plain loads, 1 bulk copies, sites per
// consumer thread); index = tile_id.
constexpr int kVariantCols = 7;
// D3Q19 rows of the split step: 16 x 8 columns, 4 resident CTAs, no producer warps.
constexpr bool split_row(const int* t) {
    return t[0] == 16 && t[1] == 8 && t[3] == 4 && t[4] == 0 && t[5] == 0;
}
int tile_shapes_d2q9(int (*out)[kVariantCols], int max);
int tile_shapes_d3q19(int (*out)[kVariantCols], int max);

cudaError_t launch_step_d2q9(int coupling, int fp32, const StepLaunch& a, cudaStream_t st);
cudaError_t launch_step_d3q19(int coupling, int fp32, const StepLaunch& a, cudaStream_t st);

cudaError_t launch_init_feq_d2q9(int coupling, int fp32, const SysDev* sys, const int4* items, int n_items,
                                 const double* d, const double* dbar, void* fbuf, cudaStream_t st);
cudaError_t launch_init_feq_d3q19(int coupling, int fp32, const SysDev* sys, const int4* items, int n_items,
                                  const double* d, const double* dbar, void* fbuf, cudaStream_t st);
// Populations i0 .. i0 + ni - 1 of one system, [population][site] in out / in.
cudaError_t launch_gather_d2q9(int fp32, const SysDev* sys, int s, int i0, int ni, int64_t n, const void* fbuf, double* out,
                               cudaStream_t st);
cudaError_t launch_gather_d3q19(int fp32, const SysDev* sys, int s, int i0, int ni, int64_t n, const void* fbuf, double* out,
                                cudaStream_t st);
cudaError_t launch_scatter_d2q9(int fp32, const SysDev* sys, int s, int i0, int ni, int64_t n, const double* in, void* fbuf,
                                cudaStream_t st);
cudaError_t launch_scatter_d3q19(int fp32, const SysDev* sys, int s, int i0, int ni, int64_t n, const double* in, void* fbuf,
                                 cudaStream_t st);
// jout (nullable): momentum field j_a at jout + a * jstride.
cudaError_t launch_obs_site_d2q9(int fp32, const SysDev* sys, const int4* items, int n_items, const void* fbuf,
                                 double* d, double* partial, double* jout, int64_t jstride, cudaStream_t st);
cudaError_t launch_obs_site_d3q19(int fp32, const SysDev* sys, const int4* items, int n_items, const void* fbuf,
                                  double* d, double* partial, double* jout, int64_t jstride, cudaStream_t st);

// ---- lattice-independent (obs.cu) ----------------------------------------
struct SysSpan {            // items [first, first + count) of one system
    int first, count;
};

// One block level of one system, as the observable kernels see it.
struct LevelDev {
    int32_t sys;
    int32_t bx, by, bz;     // block dims
    int32_t gx, gy, gz;     // blocks per axis
    int32_t child;          // index of the next finer pyramid level (-1 at the bottom)
    int64_t nblocks;
    int64_t off;            // offset of this level's block sums in the S/E arrays (-1: unit level)
    int32_t rec_first;      // records of this level in the partial-record array
    int32_t rec_count;
};

struct ObsItem {            // a range of blocks of one level
    int32_t level;          // index into the LevelDev array
    int32_t unit_level;     // bottom items also feed the separate single-site level (-1: none)
    int64_t b0, b1;
    int32_t rec, rec2;      // partial records written (rec2 for the unit level)
};

struct ObsPart {            // bottom blocks [b0, b1) of one level, sites [i0, i1) of each
    int32_t level, unit_level;
    int32_t b0, b1;         // more than one block: whole blocks, one warp each
    int32_t i0, i1;         // range of the block's sites in (x, y, z) order
    int32_t part;           // >= 0: the block has several ranges, this range's sums go there
    int32_t rec, rec2;      // records of the level (part < 0) and of the single-site level
};

struct ObsBlocks {          // bottom blocks [b0, b1) made of per_block parts each
    int32_t level, b0, b1, part0, per_block, rec;
};

struct ObsTop {             // levels of one system: top - 1 .. 0 by the top kernel, the others have records
    int32_t lv_first, n_levels, top;
};

// Order-parameter histograms: per level (nbins + 2) counts [under, bins, over]
// at counts + level * (nbins + 2); nbins = 0 disables them.
struct HistDev {
    unsigned long long* counts;
    int32_t nbins;
    double lo, inv_w;       // bin of m: floor((m - lo) * inv_w), inv_w = nbins / (hi - lo)
};

// OR status bits into the device status word (fault injection).
cudaError_t launch_set_status(int* status, int bits, cudaStream_t st);
// One CTA whose bounded wait on a barrier nothing arrives at must time out.
cudaError_t launch_selftest_wait(int* status, cudaStream_t st);

cudaError_t launch_init_noise(const SysDev* sys, const int4* items, int n_items, double amp, double* d,
                              double* partial, cudaStream_t st);
// dbar[2 s], dbar[2 s + 1]: mean density deviation of system s and 1 / its mean density.
cudaError_t launch_reduce_globals(const SysDev* sys, const SysSpan* spans, int n_sys, const double* partial,
                                  double* dbar, double* glob, int set_mass0, int count_sample, cudaStream_t st);
cudaError_t launch_set_dbar(const SysDev* sys, int n_sys, double* dbar, cudaStream_t st);
cudaError_t launch_pyr_bottom(const SysDev* sys, const LevelDev* lv, const ObsItem* items, int n_items,
                              const double* d, const double* dbar, double* S, double* E, double* rec,
                              const HistDev& hist, cudaStream_t st);
cudaError_t launch_pyr_part(const SysDev* sys, const LevelDev* lv, const ObsPart* items, int n_items,
                            const double* d, const double* dbar, double* S, double* E, double2* parts, double* rec,
                            const HistDev& hist, cudaStream_t st);
cudaError_t launch_pyr_blocks(const LevelDev* lv, const ObsBlocks* items, int n_items, const double2* parts,
                              double* S, double* E, double* rec, const HistDev& hist, cudaStream_t st);
cudaError_t launch_pyr_up(const LevelDev* lv, const ObsItem* items, int n_items, int dims3,
                          double* S, double* E, double* rec, const HistDev& hist, cudaStream_t st);
cudaError_t launch_pyr_top(const LevelDev* lv, const ObsTop* tops, int n_sys, int dims3, double* S, double* E,
                           const double* rec, double* acc, int* status, const HistDev& hist, cudaStream_t st);
cudaError_t launch_obs_accum(const LevelDev* lv, int n_levels, const double* rec, double* acc, int* status,
                             cudaStream_t st);
cudaError_t launch_advance(int64_t* step, int64_t n, cudaStream_t st);

constexpr int OBS_THREADS = 256;
constexpr int BLOCKS_PER_THREAD = 4;
constexpr int TOP_THREADS = 512;        // pyr_top_kernel: one CTA per system
// Bottom blocks of more than kThreadSites sites take a warp or a CTA instead of
// a thread (a thread's sites are a serial chain of row loads), those of more
// than kWarpSites a CTA, in ranges of kPartSites sites (16 per thread).
constexpr int kThreadSites = 32, kWarpSites = 1024, kPartSites = 4096;
// Levels of at most this many blocks go to the top kernel.  Its one CTA per
// system has one SM's FP64 unit (two operations per clock): 4,096 blocks cost
// it 30 us, 512 blocks 4 us, about a launch.
constexpr int kTopBlocks = 512;
constexpr int kMaxObsLevels = 40;       // block levels of a system (halvings of a side below 2^31, and single sites)
constexpr int REC = 6;      // per record: sum m, m^2, |m|, m^4, e, e^2

}  // namespace lbf

namespace lbf {

// ---- structure factor (Eq. 80) -------------------------------------------------
struct SkSys {             // per system: sides, twiddle-table offsets, site offset
    int32_t nx, ny, nz;
    int32_t tw_x, tw_y, tw_z;   // offsets of W_n^j = exp(-2 pi i j / n) tables (complex)
    int64_t site_offset;
    int64_t half_offset;        // first value of the system's half spectrum (kx <= nx/2)
    double inv_n;               // 1 / sites
};

cudaError_t launch_sk_twiddles(double* tw, const int* sides, const int* offs, int n_tables, int max_n,
                               cudaStream_t st);
// x pass (real phi -> complex), then y and z passes (complex -> complex), then accumulate |F|^2 / N.
cudaError_t launch_sk_x(const SkSys* sk, const int4* items, int n_items, const double* d,
                        const double* dbar, const double* tw, double* out, cudaStream_t st);
cudaError_t launch_sk_pass(const SkSys* sk, const int4* items, int n_items, int axis, const double* tw,
                           const double* in, double* out, cudaStream_t st);
// Line FFTs of every field of a sample and accumulation of its spectra, for
// systems with sides up to kSkFftMaxElems (see sk.cu).  Work lists in `items`:
// n_x items (system, first line, count, field) of the x pass, n_y of the y pass
// (3-D only), n_last (system, first line, count, 0) of the last pass; max_* are
// the largest line count x line length of an item, in complex values (of all
// fields in the last pass).
constexpr int kSkFftMaxElems = 2048;
constexpr int FFT_THREADS = 128;
bool sk_fft_side(int n);
struct FftLaunch {
    const SkSys* sk;
    const int4* items;
    int n_x, n_y, n_last, max_x, max_y, max_last;
    int dims, nf;               // fields: phi, then the momentum components (nf = 1: phi alone)
    const double *d, *dbar, *j; // j_a at j + a n_sites
    const double* tw;
    double* F;                  // half spectra, field f at F + 2 f fstride
    int64_t fstride, n_sites;
    double *acc, *jacc;         // accumulated spectra (jacc: three, n_sites apart)
};
cudaError_t launch_sk_fft(const FftLaunch& a, cudaStream_t st);
cudaError_t launch_sk_accum(const SkSys* sk, const int4* items, int n_items, const double* F, double* acc,
                            cudaStream_t st);
// Momentum spectra (see sk.cu): accumulate the x, longitudinal and transverse
// spectra of the transforms F0..F2 (F2 unused in 2-D) into acc + c * stride.
cudaError_t launch_jk_accum(const SkSys* sk, const int4* items, int n_items, int dims, const double* F0,
                            const double* F1, const double* F2, double* acc, int64_t stride, cudaStream_t st);
// Guo variant: lap = Laplacian of d, then j_a += kappa rho d_a(lap) / 2 (j at jf + a * stride).
cudaError_t launch_jk_guo_force(int lattice, const SysDev* sys, const int4* items, int n_items, const double* d,
                                double* lap, double* jf, int64_t stride, cudaStream_t st);
// Shell sums (and point counts) of nspec spectra of one system, `stride` apart: [spectrum][shell].
cudaError_t launch_sk_bin(const SkSys* sk, int sys, const double* acc, int64_t stride, int nspec, int nbins,
                          double* sums, double* counts, cudaStream_t st);

}  // namespace lbf

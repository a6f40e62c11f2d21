// Lattice-independent kernels: initial density perturbation, per-system FP64
// reductions, and the block-observable pyramid (Eqs. 46-50).
//
// The pyramid: block levels are L = S/2^i (i = 0..imax); the bottom level's
// block sums of phi and phi^2 are taken from the sites, every coarser level
// sums the 2^d children of the next finer one.  Per block the nonlinear terms
// m, m^2, |m|, m^4, E, E^2 (m = sum phi / V, E = sum phi^2 / 2V) are formed and
// reduced per item into a record; one warp per level then sums its records
// into the FP64 accumulators.  Every sum has a fixed order.
//
// Who sums what (launches of one sample, each skipped when empty):
//   pyr_bottom_kernel  bottom levels of small blocks: one thread per block
//   pyr_part_kernel    bottom levels of larger blocks (sides whose odd factor
//                      is not small): a warp per block, or a CTA per range of
//                      up to kPartSites sites of a block; with one thread per
//                      block an odd-sided system was a serial sum over all its
//                      sites (57.6 ms a sample for 32 systems of up to 141,000
//                      sites; 0.1 ms with this kernel)
//   pyr_blocks_kernel  bottom levels whose blocks have several ranges
//   pyr_up_kernel      coarser levels of more than kTopBlocks blocks
//   pyr_top_kernel     one CTA per system: its remaining coarser levels, one
//                      after another behind CTA barriers (a launch per level
//                      before: these levels are microseconds of latency each),
//                      and the sums of the records the kernels above wrote
#include "../../include/lbfluct.h"
#include "lattice_kernels.cuh"
#include "lb_launch.h"

namespace lbf {

namespace {

// Histogram counts are dynamic shared memory beside the kernels' own, together
// within what a launch gets without asking for more.
constexpr size_t kPlainShared = 48 * 1024;
constexpr size_t hist_shared(int nbins, int levels) { return sizeof(unsigned) * levels * size_t(nbins + 2); }
static_assert(sizeof(BlockSum<REC, OBS_THREADS>) + hist_shared(LB_MAX_HIST_BINS, 2) <= kPlainShared,
              "pyr_bottom_kernel, pyr_part_kernel, pyr_up_kernel");

__global__ void __launch_bounds__(AUX_THREADS)
    init_noise_kernel(const SysDev* __restrict__ sysv, const int4* __restrict__ items, double amp,
                      double* __restrict__ d, double* __restrict__ partial) {
    __shared__ BlockSum<1, AUX_THREADS> sh;
    const int4 it = items[blockIdx.x];
    const SysDev& S = sysv[it.x];
    double acc[1] = {0.0};
    for (int j = 0; j < SITES_PER_THREAD; ++j) {
        const int site = it.y + j * AUX_THREADS + threadIdx.x;
        if (site >= it.z) break;
        const uint4 w = site_draw(S, uint32_t(site), 0, 0xFFu);
        const double u = (double(w.x) + 0.5) * 2.3283064365386962890625e-10;
        const double v = amp * (2.0 * u - 1.0);
        d[S.site_offset + site] = v;
        acc[0] += v;
    }
    block_sum(acc, sh);
    if (threadIdx.x == 0) partial[int64_t(blockIdx.x) * 4] = acc[0];
}

// Per system: the sums over its items of partial[item * 4 + (0..3)] in a fixed
// order (sum d, sum jx, sum jy, sum jz), then the mean deviation and the
// global bookkeeping.  glob layout per system (8 doubles): n_samples, mass0,
// mass, jx, jy, jz, rho_mean, spare.
__global__ void __launch_bounds__(AUX_THREADS)
    reduce_globals_kernel(const SysDev* __restrict__ sysv, const SysSpan* __restrict__ spans,
                          const double* __restrict__ partial, double* __restrict__ dbar, double* __restrict__ glob,
                          int set_mass0, int count_sample) {
    __shared__ BlockSum<4, AUX_THREADS> sh;
    const int s = blockIdx.x;
    const SysSpan sp = spans[s];
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int it = threadIdx.x; it < sp.count; it += AUX_THREADS) {
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] += partial[int64_t(sp.first + it) * 4 + k];
    }
    block_sum(acc, sh);
    if (threadIdx.x != 0) return;
    const SysDev& S = sysv[s];
    const double n = double(S.n_sites);
    const double mass = S.rho_c * n + acc[0];
    dbar[2 * s] = acc[0] / n;
    dbar[2 * s + 1] = 1.0 / (S.rho_c + acc[0] / n);
    double* g = glob + s * 8;
    if (set_mass0) {
        g[0] = 0.0;
        g[1] = mass;
    }
    if (count_sample) g[0] += 1.0;
    g[2] = mass;
    g[3] = acc[1];
    g[4] = acc[2];
    g[5] = acc[3];
    g[6] = mass / n;
}

__global__ void set_dbar_kernel(const SysDev* __restrict__ sysv, int n_sys, double* __restrict__ dbar) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < n_sys) dbar[2 * s] = sysv[s].rho_c;
}

// Terms of blocks of volume V from their sums s of phi and e of phi^2: t
// collects the sums of s, s^2, |s|, s^4, e, e^2, and finish_terms turns them
// into those of m = s / V, m^2, |m|, m^4, E = e / 2V, E^2.
__device__ __forceinline__ void add_terms(double (&t)[REC], double s, double e) {
    const double s2 = s * s;
    t[0] += s;
    t[1] += s2;
    t[2] += fabs(s);
    t[3] += s2 * s2;
    t[4] += e;
    t[5] += e * e;
}
__device__ __forceinline__ void finish_terms(double (&t)[REC], double inv_v) {
    const double v2 = inv_v * inv_v, h = 0.5 * inv_v;
    t[0] *= inv_v;
    t[1] *= v2;
    t[2] *= inv_v;
    t[3] *= v2 * v2;
    t[4] *= h;
    t[5] *= h * h;
}

// The same for single sites (V = 1, e = s^2: its sums are halves and quarters
// of those of m^2 and m^4): t = sum m, m^2, |m|, m^4.
__device__ __forceinline__ void add_site_terms(double (&t)[REC], double m, double m2) {
    t[0] += m;
    t[1] += m2;
    t[2] += fabs(m);
    t[3] += m2 * m2;
}
__device__ __forceinline__ void finish_site_terms(double (&t)[REC]) {
    t[4] = 0.5 * t[1];
    t[5] = 0.25 * t[3];
}

// Histogram bin of a block value m: 1 + floor(t), t = (m - lo) * inv_w, with
// 0 below the range and nbins + 1 at or above it (and for NaN).  The product
// is formed from the rounded difference, as in the plain definition.
__device__ __forceinline__ int hist_bin(double m, const HistDev& H) {
    const double t = __dmul_rn(__dsub_rn(m, H.lo), H.inv_w);
    if (t >= 0.0) return t < double(H.nbins) ? 1 + int(t) : H.nbins + 1;
    return t < 0.0 ? 0 : H.nbins + 1;
}

// Per-CTA histograms in shared memory (32-bit counts; a CTA sees far fewer
// than 2^32 values), added to the 64-bit global counts at the end.
__device__ __forceinline__ void hist_clear(unsigned* sh, int n) {
    for (int k = threadIdx.x; k < n; k += blockDim.x) sh[k] = 0u;
}
__device__ __forceinline__ void hist_flush(const unsigned* sh, int n, unsigned long long* g) {
    for (int k = threadIdx.x; k < n; k += blockDim.x)
        if (sh[k]) atomicAdd(g + k, (unsigned long long)sh[k]);
}

__device__ __forceinline__ double block_volume(const LevelDev& lv) { return double(lv.bx) * lv.by * lv.bz; }

// The CTA's sums of a level's terms as a record (a division occupies the FP64
// unit like ten additions: one thread's, not every thread's).
__device__ __forceinline__ void block_record(double (&t)[REC], const LevelDev& lv, BlockSum<REC, OBS_THREADS>& sh,
                                             double* rec) {
    block_sum(t, sh);
    if (threadIdx.x != 0) return;
    finish_terms(t, 1.0 / block_volume(lv));
    for (int k = 0; k < REC; ++k) rec[k] = t[k];
}
__device__ __forceinline__ void site_record(double (&t)[REC], BlockSum<4, OBS_THREADS>& sh, double* rec) {
    double v[4] = {t[0], t[1], t[2], t[3]};
    block_sum(v, sh);
    if (threadIdx.x != 0) return;
    for (int k = 0; k < 4; ++k) t[k] = v[k];
    finish_site_terms(t);
    for (int k = 0; k < REC; ++k) rec[k] = t[k];
}

// Block coordinates of block b of a pyramid level: 2^k blocks per axis.
__device__ __forceinline__ void block_coords(const LevelDev& lv, int b, int& X, int& Y, int& Z) {
    const int kx = 31 - __clz(lv.gx), ky = 31 - __clz(lv.gy);
    X = b & (lv.gx - 1);
    Y = (b >> kx) & (lv.gy - 1);
    Z = b >> (kx + ky);
}

// Bottom pyramid level: block sums of phi, phi^2 straight from the sites; the
// separate single-site level (if any) is fed from the same loop.  With
// histograms on, each block value m (and each site value of the single-site
// level) is also binned.
__global__ void __launch_bounds__(OBS_THREADS)
    pyr_bottom_kernel(const SysDev* __restrict__ sysv, const LevelDev* __restrict__ lvv,
                      const ObsItem* __restrict__ items, const double* __restrict__ d,
                      const double* __restrict__ dbar, double* __restrict__ Sg, double* __restrict__ Eg,
                      double* __restrict__ rec, const HistDev H) {
    __shared__ BlockSum<REC, OBS_THREADS> sh;
    auto& sh4 = reinterpret_cast<BlockSum<4, OBS_THREADS>&>(sh);   // never between sh's barriers
    extern __shared__ unsigned shist[];          // [block level | single-site level], nbins + 2 each
    const ObsItem it = items[blockIdx.x];
    const LevelDev lv = lvv[it.level];
    const SysDev& S = sysv[lv.sys];
    const double* ds = d + S.site_offset;
    const double db = dbar[2 * lv.sys], inv_rbar = dbar[2 * lv.sys + 1];
    const int nh = H.nbins + 2;
    const bool hist = H.nbins > 0;
    const double inv_v = hist ? 1.0 / block_volume(lv) : 0.0;
    const bool hist_u = hist && it.unit_level >= 0;
    if (hist) {
        hist_clear(shist, hist_u ? 2 * nh : nh);
        __syncthreads();
    }
    double tb[REC] = {0, 0, 0, 0, 0, 0};
    double tu[REC] = {0, 0, 0, 0, 0, 0};
    const int nx = S.nx, ny = S.ny;
    const bool sites = lv.bx == 1 && lv.by == 1 && lv.bz == 1;   // blocks are the sites, in site order
    for (int b = int(it.b0) + threadIdx.x; b < int(it.b1); b += OBS_THREADS) {
        double s = 0.0, e = 0.0;
        if (sites) {
            s = (ds[b] - db) * inv_rbar;
            e = s * s;
        } else {
            int X, Y, Z;
            block_coords(lv, b, X, Y, Z);
            for (int z = 0; z < lv.bz; ++z)
                for (int y = 0; y < lv.by; ++y) {
                    const int row = X * lv.bx + nx * (Y * lv.by + y + ny * (Z * lv.bz + z));
                    for (int x = 0; x < lv.bx; ++x) {
                        const double phi = (ds[row + x] - db) * inv_rbar;
                        s += phi;
                        e += phi * phi;
                        if (it.unit_level >= 0) add_site_terms(tu, phi, phi * phi);
                        if (hist_u) atomicAdd(shist + nh + hist_bin(phi, H), 1u);
                    }
                }
        }
        Sg[lv.off + b] = s;
        Eg[lv.off + b] = e;
        if (sites) add_site_terms(tb, s, e);
        else add_terms(tb, s, e);
        if (hist) atomicAdd(shist + hist_bin(s * inv_v, H), 1u);
    }
    // (of single sites the last two sums follow from the others)
    if (sites) site_record(tb, sh4, rec + int64_t(it.rec) * REC);
    else block_record(tb, lv, sh, rec + int64_t(it.rec) * REC);
    if (it.unit_level >= 0) site_record(tu, sh4, rec + int64_t(it.rec2) * REC);
    if (hist) {
        __syncthreads();
        hist_flush(shist, nh, H.counts + int64_t(it.level) * nh);
        if (hist_u) hist_flush(shist + nh, nh, H.counts + int64_t(it.unit_level) * nh);
    }
}

// Bottom level of blocks too large for one thread each.  Items either hold
// several whole blocks, one warp each (warp w takes blocks b0 + w, b0 + w + 8,
// ...), or a range [i0, i1) of one block's sites, summed by the whole CTA: then
// the block is complete when the range is all of it (part < 0), else the CTA
// leaves its sums of phi and phi^2 in parts[part] for pyr_blocks_kernel.
__global__ void __launch_bounds__(OBS_THREADS)
    pyr_part_kernel(const SysDev* __restrict__ sysv, const LevelDev* __restrict__ lvv,
                    const ObsPart* __restrict__ items, const double* __restrict__ d, const double* __restrict__ dbar,
                    double* __restrict__ Sg, double* __restrict__ Eg, double2* __restrict__ parts,
                    double* __restrict__ rec, const HistDev H) {
    constexpr int NW = OBS_THREADS / 32;
    __shared__ BlockSum<REC, OBS_THREADS> sh;
    auto& sh4 = reinterpret_cast<BlockSum<4, OBS_THREADS>&>(sh);
    auto& sh2 = reinterpret_cast<BlockSum<2, OBS_THREADS>&>(sh);   // used before sh, a barrier apart
    extern __shared__ unsigned shist[];          // [block level | single-site level], nbins + 2 each
    const ObsPart it = items[blockIdx.x];
    const LevelDev lv = lvv[it.level];
    const SysDev& S = sysv[lv.sys];
    const double* ds = d + S.site_offset;
    const double db = dbar[2 * lv.sys], inv_rbar = dbar[2 * lv.sys + 1];
    const int nh = H.nbins + 2;
    const bool hist = H.nbins > 0;
    const double inv_v = hist ? 1.0 / block_volume(lv) : 0.0;
    if (hist) {
        hist_clear(shist, 2 * nh);
        __syncthreads();
    }
    double tb[REC] = {0, 0, 0, 0, 0, 0};
    double tu[REC] = {0, 0, 0, 0, 0, 0};
    const int nx = S.nx, ny = S.ny;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool by_warp = it.b1 - it.b0 > 1;
    const int step = by_warp ? 32 : OBS_THREADS;
    auto block_done = [&](int b, double s, double e) {
        Sg[lv.off + b] = s;
        Eg[lv.off + b] = e;
        add_terms(tb, s, e);
        if (hist) atomicAdd(shist + hist_bin(s * inv_v, H), 1u);
    };
    for (int b = it.b0 + (by_warp ? warp : 0); b < it.b1; b += by_warp ? NW : 1) {
        int X, Y, Z;
        block_coords(lv, b, X, Y, Z);
        const double* corner = ds + (X * lv.bx + nx * (Y * lv.by + int64_t(ny) * (Z * lv.bz)));
        double v[2] = {0.0, 0.0};
        for (int i = it.i0 + (by_warp ? lane : int(threadIdx.x)); i < it.i1; i += step) {
            const int r = i / lv.bx, x = i - r * lv.bx, z = r / lv.by, y = r - z * lv.by;
            const double phi = (corner[x + nx * (y + int64_t(ny) * z)] - db) * inv_rbar;
            v[0] += phi;
            v[1] += phi * phi;
            add_site_terms(tu, phi, phi * phi);
            if (hist) atomicAdd(shist + nh + hist_bin(phi, H), 1u);
        }
        if (by_warp) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                v[0] += __shfl_down_sync(0xffffffffu, v[0], o);
                v[1] += __shfl_down_sync(0xffffffffu, v[1], o);
            }
            if (lane == 0) block_done(b, v[0], v[1]);
        } else {
            block_sum(v, sh2);
            if (threadIdx.x == 0) {
                if (it.part < 0) block_done(b, v[0], v[1]);
                else parts[it.part] = make_double2(v[0], v[1]);
            }
            __syncthreads();
        }
    }
    if (it.part < 0) block_record(tb, lv, sh, rec + int64_t(it.rec) * REC);
    site_record(tu, sh4, rec + int64_t(it.rec2) * REC);
    if (hist) {
        __syncthreads();
        if (it.part < 0) hist_flush(shist, nh, H.counts + int64_t(it.level) * nh);
        hist_flush(shist + nh, nh, H.counts + int64_t(it.unit_level) * nh);
    }
}

// Blocks of several ranges: one warp per block sums its parts (parts of a
// block are consecutive, part0 + b * per_block on).
__global__ void __launch_bounds__(OBS_THREADS)
    pyr_blocks_kernel(const LevelDev* __restrict__ lvv, const ObsBlocks* __restrict__ items,
                      const double2* __restrict__ parts, double* __restrict__ Sg, double* __restrict__ Eg,
                      double* __restrict__ rec, const HistDev H) {
    constexpr int NW = OBS_THREADS / 32;
    __shared__ BlockSum<REC, OBS_THREADS> sh;
    const ObsBlocks it = items[blockIdx.x];
    const LevelDev lv = lvv[it.level];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double tb[REC] = {0, 0, 0, 0, 0, 0};
    for (int b = it.b0 + warp; b < it.b1; b += NW) {
        const double2* p = parts + it.part0 + int64_t(b) * it.per_block;
        double s = 0.0, e = 0.0;
        for (int k = lane; k < it.per_block; k += 32) {
            const double2 v = p[k];
            s += v.x;
            e += v.y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_down_sync(0xffffffffu, s, o);
            e += __shfl_down_sync(0xffffffffu, e, o);
        }
        if (lane == 0) {
            Sg[lv.off + b] = s;
            Eg[lv.off + b] = e;
            add_terms(tb, s, e);
            if (H.nbins > 0)
                atomicAdd(H.counts + int64_t(it.level) * (H.nbins + 2) + hist_bin(s * (1.0 / block_volume(lv)), H), 1ull);
        }
    }
    block_record(tb, lv, sh, rec + int64_t(it.rec) * REC);
}

// Sums of phi and phi^2 of block b of level lv over its 2^d children (level
// ch), in the order x, y, z.
__device__ __forceinline__ void children_sum(const LevelDev& lv, const LevelDev& ch, int b, int dims3,
                                             const double* Sg, const double* Eg, double& s, double& e) {
    int X, Y, Z;
    block_coords(lv, b, X, Y, Z);
    s = e = 0.0;
    const int nz = dims3 ? 2 : 1;
    for (int dz = 0; dz < nz; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const int64_t c = ch.off + 2 * X + ch.gx * (2 * Y + dy + int64_t(ch.gy) * (nz * Z + dz));
            s += Sg[c];
            e += Eg[c];
            s += Sg[c + 1];
            e += Eg[c + 1];
        }
}

// One coarser level: each block sums its 2^d children of the next finer level.
__global__ void __launch_bounds__(OBS_THREADS)
    pyr_up_kernel(const LevelDev* __restrict__ lvv, const ObsItem* __restrict__ items, int dims3,
                  double* __restrict__ Sg, double* __restrict__ Eg, double* __restrict__ rec, const HistDev H) {
    __shared__ BlockSum<REC, OBS_THREADS> sh;
    extern __shared__ unsigned shist[];
    const ObsItem it = items[blockIdx.x];
    const LevelDev lv = lvv[it.level];
    const LevelDev ch = lvv[lv.child];
    const int nh = H.nbins + 2;
    const bool hist = H.nbins > 0;
    const double inv_v = hist ? 1.0 / block_volume(lv) : 0.0;
    if (hist) {
        hist_clear(shist, nh);
        __syncthreads();
    }
    double tb[REC] = {0, 0, 0, 0, 0, 0};
    for (int b = int(it.b0) + threadIdx.x; b < int(it.b1); b += OBS_THREADS) {
        double s, e;
        children_sum(lv, ch, b, dims3, Sg, Eg, s, e);
        Sg[lv.off + b] = s;
        Eg[lv.off + b] = e;
        add_terms(tb, s, e);
        if (hist) atomicAdd(shist + hist_bin(s * inv_v, H), 1u);
    }
    block_record(tb, lv, sh, rec + int64_t(it.rec) * REC);
    if (hist) {
        __syncthreads();
        hist_flush(shist, nh, H.counts + int64_t(it.level) * nh);
    }
}

// acc layout per level (7 doubles): n, sum m, m^2, |m|, m^4, e, e^2
__device__ __forceinline__ void accumulate_level(double* a, double nblocks, const double (&t)[REC], int* status) {
    a[0] += nblocks;
    bool finite = true;
    for (int k = 0; k < REC; ++k) {
        a[1 + k] += t[k];
        finite = finite && isfinite(t[k]);
    }
    if (!finite) atomicOr(status, ST_NONFINITE);
}

// One warp: the records of a level, summed by lanes 32 apart and a shuffle
// tree, into its accumulators.  (One thread in order before: 0.1 ms of
// dependent loads for the 256 records of a 64^3 system.)
__device__ __forceinline__ void accumulate_records(const LevelDev& lv, const double* __restrict__ rec, double* a,
                                                   int* status) {
    const int lane = threadIdx.x & 31;
    double t[REC] = {0, 0, 0, 0, 0, 0};
    for (int r = lane; r < lv.rec_count; r += 32)
#pragma unroll
        for (int k = 0; k < REC; ++k) t[k] += rec[int64_t(lv.rec_first + r) * REC + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < REC; ++k) t[k] += __shfl_down_sync(0xffffffffu, t[k], o);
    if (lane == 0) accumulate_level(a, double(lv.nblocks), t, status);
}

// Block sums of alternate levels: the first has up to kTopBlocks blocks, every
// next one at most a quarter of the one below it.
template <int NC>
struct TopShared {
    BlockSum<REC, NC> sh;
    double bs0[kTopBlocks], be0[kTopBlocks], bs1[kTopBlocks / 4], be1[kTopBlocks / 4];
    double sums[kMaxObsLevels][REC];
    LevelDev lvs[kMaxObsLevels];
};
static_assert(sizeof(TopShared<TOP_THREADS / 2>) + hist_shared(LB_MAX_HIST_BINS, 1) <= kPlainShared, "pyr_top_kernel");

// The coarsest levels of one system per CTA: levels top - 1 .. 0 (level `top`
// is complete), one after another in the first kTopChain threads, with the
// block sums of the level below in shared memory (the first takes them from
// memory) and levels of at most 32 blocks in one warp without a barrier; the
// levels' sums are accumulated together at the end.  The other warps meanwhile
// accumulate the records of the other levels.  A chain of latencies: 16^3, four
// levels, 17 us (22 us with the block sums in memory and CTA-wide barriers).
__global__ void __launch_bounds__(TOP_THREADS)
    pyr_top_kernel(const LevelDev* __restrict__ lvv, const ObsTop* __restrict__ tops, int dims3, double* Sg,
                   double* Eg, const double* __restrict__ rec, double* __restrict__ acc, int* status,
                   const HistDev H) {
    constexpr int NC = TOP_THREADS / 2;
    __shared__ TopShared<NC> sm;
    auto& sh = sm.sh;
    auto& sums = sm.sums;
    auto& lvs = sm.lvs;
    extern __shared__ unsigned shist[];
    const ObsTop T = tops[blockIdx.x];
    const int nh = H.nbins + 2, tid = threadIdx.x;
    const bool hist = H.nbins > 0;
    for (int l = tid; l < T.n_levels; l += TOP_THREADS) lvs[l] = lvv[T.lv_first + l];
    __syncthreads();
    double* const my_acc = acc + int64_t(T.lv_first) * 7;
    if (tid >= NC) {
        for (int l = T.top + (tid - NC) / 32; l < T.n_levels; l += NC / 32)
            accumulate_records(lvs[l], rec, my_acc + 7 * l, status);
        return;
    }
    for (int l = T.top - 1; l >= 0; --l) {
        const LevelDev& lv = lvs[l];
        const LevelDev& ch = lvs[l + 1];
        const int nb = int(lv.nblocks), dst = (T.top - 1 - l) & 1;       // (0: the first level, the largest)
        double* const bs = dst ? sm.bs1 : sm.bs0;
        double* const be = dst ? sm.be1 : sm.be0;
        const double* const cs = dst ? sm.bs0 : sm.bs1;                  // the level below
        const double* const ce = dst ? sm.be0 : sm.be1;
        const double inv_v = hist ? 1.0 / block_volume(lv) : 0.0;
        const bool warp_only = nb <= 32;
        if (warp_only && tid >= 32) break;                // the remaining levels have no more blocks than this one
        if (hist) {
            for (int k = tid; k < nh; k += warp_only ? 32 : NC) shist[k] = 0u;
            if (warp_only) __syncwarp();
            else named_barrier(1, NC);
        }
        double tb[REC] = {0, 0, 0, 0, 0, 0};
        for (int b = tid; b < nb; b += NC) {
            double s = 0.0, e = 0.0;
            if (l == T.top - 1) {
                children_sum(lv, ch, b, dims3, Sg, Eg, s, e);
            } else {
                int X, Y, Z;
                block_coords(lv, b, X, Y, Z);
                const int nz = dims3 ? 2 : 1;
                for (int dz = 0; dz < nz; ++dz)
#pragma unroll
                    for (int dy = 0; dy < 2; ++dy) {
                        const int c = 2 * X + ch.gx * (2 * Y + dy + ch.gy * (nz * Z + dz));
                        s += cs[c];
                        e += ce[c];
                        s += cs[c + 1];
                        e += ce[c + 1];
                    }
            }
            bs[b] = s;
            be[b] = e;
            add_terms(tb, s, e);
            if (hist) atomicAdd(shist + hist_bin(s * inv_v, H), 1u);
        }
        if (warp_only) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int k = 0; k < REC; ++k) tb[k] += __shfl_down_sync(0xffffffffu, tb[k], o);
        } else {
            block_sum<REC, NC, 1>(tb, sh, min(NC, nb));   // its barriers also order this level's block sums
        }
        if (tid == 0) {
#pragma unroll
            for (int k = 0; k < REC; ++k) sums[l][k] = tb[k];
        }
        if (hist) {
            if (warp_only) __syncwarp();
            unsigned long long* g = H.counts + int64_t(T.lv_first + l) * nh;
            for (int k = tid; k < nh; k += warp_only ? 32 : NC)
                if (shist[k]) atomicAdd(g + k, (unsigned long long)shist[k]);
        }
        if (warp_only) __syncwarp();
        else named_barrier(1, NC);
    }
    // warp 0, which has seen every level end: a lane per level adds its sums
    if (tid < T.top) {
        double t[REC];
#pragma unroll
        for (int k = 0; k < REC; ++k) t[k] = sums[tid][k];
        const LevelDev& lv = lvs[tid];
        finish_terms(t, 1.0 / block_volume(lv));
        accumulate_level(my_acc + 7 * tid, double(lv.nblocks), t, status);
    }
}

// One warp per level (the allocation-free entry point, whose levels all have records).
__global__ void obs_accum_kernel(const LevelDev* __restrict__ lvv, const double* __restrict__ rec,
                                 double* __restrict__ acc, int* status) {
    accumulate_records(lvv[blockIdx.x], rec, acc + int64_t(blockIdx.x) * 7, status);
}

__global__ void advance_kernel(int64_t* step, int64_t n) { *step += n; }

// Fault injection: OR bits into the device status word (as a kernel would on
// detecting the condition).
__global__ void set_status_kernel(int* status, int bits) { atomicOr(status, bits); }

// Self-test of the bounded waits: one CTA waits on an mbarrier that nothing
// arrives at; every thread must give up and the status must record it.
__global__ void selftest_wait_kernel(int* status) {
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
    }
    __syncthreads();
    if (mbar_wait(&bar, 0u, &abort_flag, status)) atomicOr(status, 1 << 30);   // cannot complete
}

}  // namespace

cudaError_t launch_init_noise(const SysDev* sys, const int4* items, int n_items, double amp, double* d,
                              double* partial, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    init_noise_kernel<<<n_items, AUX_THREADS, 0, st>>>(sys, items, amp, d, partial);
    return cudaGetLastError();
}

cudaError_t launch_reduce_globals(const SysDev* sys, const SysSpan* spans, int n_sys, const double* partial,
                                  double* dbar, double* glob, int set_mass0, int count_sample, cudaStream_t st) {
    reduce_globals_kernel<<<n_sys, AUX_THREADS, 0, st>>>(sys, spans, partial, dbar, glob, set_mass0, count_sample);
    return cudaGetLastError();
}

cudaError_t launch_set_dbar(const SysDev* sys, int n_sys, double* dbar, cudaStream_t st) {
    set_dbar_kernel<<<(n_sys + 127) / 128, 128, 0, st>>>(sys, n_sys, dbar);
    return cudaGetLastError();
}

cudaError_t launch_pyr_bottom(const SysDev* sys, const LevelDev* lv, const ObsItem* items, int n_items,
                              const double* d, const double* dbar, double* S, double* E, double* rec,
                              const HistDev& hist, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    const size_t shm = hist.nbins > 0 ? hist_shared(hist.nbins, 2) : 0;
    pyr_bottom_kernel<<<n_items, OBS_THREADS, shm, st>>>(sys, lv, items, d, dbar, S, E, rec, hist);
    return cudaGetLastError();
}

cudaError_t launch_pyr_part(const SysDev* sys, const LevelDev* lv, const ObsPart* items, int n_items,
                            const double* d, const double* dbar, double* S, double* E, double2* parts, double* rec,
                            const HistDev& hist, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    const size_t shm = hist.nbins > 0 ? hist_shared(hist.nbins, 2) : 0;
    pyr_part_kernel<<<n_items, OBS_THREADS, shm, st>>>(sys, lv, items, d, dbar, S, E, parts, rec, hist);
    return cudaGetLastError();
}

cudaError_t launch_pyr_blocks(const LevelDev* lv, const ObsBlocks* items, int n_items, const double2* parts,
                              double* S, double* E, double* rec, const HistDev& hist, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    pyr_blocks_kernel<<<n_items, OBS_THREADS, 0, st>>>(lv, items, parts, S, E, rec, hist);
    return cudaGetLastError();
}

cudaError_t launch_pyr_top(const LevelDev* lv, const ObsTop* tops, int n_sys, int dims3, double* S, double* E,
                           const double* rec, double* acc, int* status, const HistDev& hist, cudaStream_t st) {
    const size_t shm = hist.nbins > 0 ? hist_shared(hist.nbins, 1) : 0;
    pyr_top_kernel<<<n_sys, TOP_THREADS, shm, st>>>(lv, tops, dims3, S, E, rec, acc, status, hist);
    return cudaGetLastError();
}

cudaError_t launch_pyr_up(const LevelDev* lv, const ObsItem* items, int n_items, int dims3,
                          double* S, double* E, double* rec, const HistDev& hist, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    const size_t shm = hist.nbins > 0 ? hist_shared(hist.nbins, 1) : 0;
    pyr_up_kernel<<<n_items, OBS_THREADS, shm, st>>>(lv, items, dims3, S, E, rec, hist);
    return cudaGetLastError();
}

cudaError_t launch_obs_accum(const LevelDev* lv, int n_levels, const double* rec, double* acc, int* status,
                             cudaStream_t st) {
    obs_accum_kernel<<<n_levels, 32, 0, st>>>(lv, rec, acc, status);
    return cudaGetLastError();
}

cudaError_t launch_advance(int64_t* step, int64_t n, cudaStream_t st) {
    advance_kernel<<<1, 1, 0, st>>>(step, n);
    return cudaGetLastError();
}

cudaError_t launch_selftest_wait(int* status, cudaStream_t st) {
    selftest_wait_kernel<<<1, 64, 0, st>>>(status);
    return cudaGetLastError();
}

cudaError_t launch_set_status(int* status, int bits, cudaStream_t st) {
    set_status_kernel<<<1, 1, 0, st>>>(status, bits);
    return cudaGetLastError();
}

}  // namespace lbf

// Lattice-dependent auxiliary kernels: initial equilibrium, population
// gather/scatter for host I/O, and the per-site pass of the observables.
// All reductions are fixed-order (per thread sequential, then a warp-shuffle
// tree and a cross-warp stage), so results are bitwise reproducible run to run.
#pragma once

#include "lb_device.cuh"
#include "lb_launch.h"

namespace lbf {

// Work item of a site pass: (system, first site, end site, unused).
// Deterministic sum of K doubles over the CTA; result valid in thread 0, and
// (after its last barrier) in res.  A warp instruction occupies the FP64 unit
// for 16 cycles whatever its mask, so the sum is packed: warp k adds the warps'
// values lane by lane and reduces the 32 sums by shuffles, 12 additions per
// value instead of 5 per value and warp.  Only threads below `active` (a
// multiple of 32 or the CTA size) bring values.
template <int K, int NT>
struct BlockSum {
    static_assert(NT % 32 == 0 && NT <= 1024, "whole warps");
    double v[K][NT];
    double res[K];
};
// The NT threads are the CTA's first; BAR > 0: only they take part, on that
// named barrier.
template <int K, int NT, int BAR = 0>
__device__ __forceinline__ void block_sum(double (&v)[K], BlockSum<K, NT>& sh, int active = NT) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (active + 31) >> 5;
    auto barrier = [] {
        if constexpr (BAR > 0) named_barrier(BAR, NT);
        else __syncthreads();
    };
    if (w < nw) {
#pragma unroll
        for (int k = 0; k < K; ++k) sh.v[k][threadIdx.x] = v[k];
    }
    barrier();
    for (int k = w; k < K; k += NW) {
        double s = sh.v[k][lane];
        for (int u = 1; u < nw; ++u) s += sh.v[k][32 * u + lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) sh.res[k] = s;
    }
    barrier();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] = sh.res[k];
    }
}

__device__ __forceinline__ void site_coords(int site, int nx, int ny, int& x, int& y, int& z) {
    x = site % nx;
    const int r = site / nx;
    y = r % ny;
    z = r / ny;
}

// f = f^eq(rho, u = 0, grad rho) at every site, written to the pull layout:
// buf_i(r - c_i) = f_i(r, 0).  rho = rho_c + d - dbar (d in FP64 scratch).
template <class L, int CP, class Real>
__global__ void __launch_bounds__(AUX_THREADS)
    init_feq_kernel(const SysDev* __restrict__ sysv, const int4* __restrict__ items, const double* __restrict__ d,
                    const double* __restrict__ dbar, Real* __restrict__ fbuf) {
    const int4 it = items[blockIdx.x];
    const SysDev& S = sysv[it.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz;
    const int64_t N = S.n_sites;
    const double* ds = d + S.site_offset;
    const double db = dbar[2 * it.x];
    for (int j = 0; j < SITES_PER_THREAD; ++j) {
        const int site = it.y + j * AUX_THREADS + threadIdx.x;
        if (site >= it.z) break;
        int x, y, z;
        site_coords(site, nx, ny, x, y, z);
        // wrapped neighbour coordinates x + d (d = -1, 0, 1) and their offsets
        const int X[3] = {wrap1(x - 1, nx), x, wrap1(x + 1, nx)};
        const int Y[3] = {wrap1(y - 1, ny) * nx, y * nx, wrap1(y + 1, ny) * nx};
        const int Z[3] = {L::D == 3 ? wrap1(z - 1, nz) * nx * ny : 0, z * nx * ny,
                          L::D == 3 ? wrap1(z + 1, nz) * nx * ny : 0};
        auto nb = [&](int i) { return ds[X[1 + L::c(i, 0)] + Y[1 + L::c(i, 1)] + Z[1 + L::c(i, 2)]] - db; };
        const double drho = ds[site] - db;
        const double rho = S.rho_c + drho;
        const double phi = drho * S.inv_rho_c;
        const double df0 = phi * (S.a + S.b * phi * phi);
        const double f0 = phi * phi * (0.5 * S.a + 0.25 * S.b * phi * phi);
        const double p0 = rho * S.inv_rho_c * df0 - f0;
        double feq[L::Q];
        double s = 0.0;
        if constexpr (CP == MODEQ && L::D == 2) {
            double gx = 0.0, gy = 0.0, lap = 0.0;
#pragma unroll
            for (int i = 1; i < L::Q; ++i) {
                const double rn = nb(i);
                gx += 3.0 * L::w(i) * L::c(i, 0) * rn;
                gy += 3.0 * L::w(i) * L::c(i, 1) * rn;
                lap += 6.0 * L::w(i) * (rn - drho);
            }
            const double iso = p0 - S.kappa * rho * lap;
#pragma unroll
            for (int i = 1; i < L::Q; ++i) {
                feq[i] = pooley_w(i) * iso +
                         S.kappa * (pooley_wxx(i) * gx * gx + pooley_wyy(i) * gy * gy + pooley_wxy(i) * gx * gy);
                s += feq[i];
            }
        } else if constexpr (CP == MODEQ) {
            // D3Q19 modified equilibrium at rest: 3 t_i iso + kappa t_i [(9/2)(c.g)^2 - (9/2) c^2 |g|^2 + (9/2)|g|^2]
            double g[3] = {0.0, 0.0, 0.0}, lap = 0.0;
#pragma unroll
            for (int i = 1; i < L::Q; ++i) {
                const double rn = nb(i);
#pragma unroll
                for (int a = 0; a < 3; ++a) g[a] += 3.0 * L::w(i) * L::c(i, a) * rn;
                lap += 6.0 * L::w(i) * (rn - drho);
            }
            const double iso = p0 - S.kappa * rho * lap;
            const double g2 = g[0] * g[0] + g[1] * g[1] + g[2] * g[2];
#pragma unroll
            for (int i = 1; i < L::Q; ++i) {
                const double cg = L::c(i, 0) * g[0] + L::c(i, 1) * g[1] + L::c(i, 2) * g[2];
                const double c2 = double(L::c(i, 0) * L::c(i, 0) + L::c(i, 1) * L::c(i, 1) + L::c(i, 2) * L::c(i, 2));
                feq[i] = 3.0 * L::w(i) * iso + S.kappa * L::w(i) * (4.5 * cg * cg - 4.5 * c2 * g2 + 4.5 * g2);
                s += feq[i];
            }
        } else {
#pragma unroll
            for (int i = 1; i < L::Q; ++i) {
                feq[i] = 3.0 * L::w(i) * p0;
                s += feq[i];
            }
        }
        feq[0] = drho - s;
#pragma unroll
        for (int i = 0; i < L::Q; ++i)
            fbuf[S.pop_offset + int64_t(i) * N + (X[1 - L::c(i, 0)] + Y[1 - L::c(i, 1)] + Z[1 - L::c(i, 2)])] =
                Real(feq[i]);
    }
}

// Element of population i that the pull of site `site` reads: buf_i(r - c_i).
template <class L>
__device__ __forceinline__ int64_t pulled_element(const SysDev& S, int site, int i) {
    int x, y, z;
    site_coords(site, S.nx, S.ny, x, y, z);
    int cx = 0, cy = 0, cz = 0;
#pragma unroll
    for (int q = 0; q < L::Q; ++q)
        if (q == i) {
            cx = L::c(q, 0);
            cy = L::c(q, 1);
            cz = L::c(q, 2);
        }
    const int sx = wrapm(x - cx, S.nx), sy = wrapm(y - cy, S.ny), sz = wrapm(z - cz, S.nz);
    return S.pop_offset + int64_t(i) * S.n_sites + (sx + S.nx * (sy + S.ny * sz));
}

// out[k][site] = f_i(r, t) = buf_i(r - c_i) + rho_c [i == 0] for the populations
// i = i0 + k, k the CTA's y index.
template <class L, class Real>
__global__ void __launch_bounds__(AUX_THREADS)
    gather_kernel(const SysDev* __restrict__ sysv, int sys, int i0, const Real* __restrict__ fbuf,
                  double* __restrict__ out) {
    const SysDev& S = sysv[sys];
    const int64_t site = int64_t(blockIdx.x) * AUX_THREADS + threadIdx.x;
    if (site >= S.n_sites) return;
    const int i = i0 + blockIdx.y;
    const double v = double(fbuf[pulled_element<L>(S, int(site), i)]);
    out[int64_t(blockIdx.y) * S.n_sites + site] = v + (i == 0 ? S.rho_c : 0.0);
}

// buf_i(r - c_i) = f_i(r) - rho_c [i == 0] for the populations i = i0 + k.
template <class L, class Real>
__global__ void __launch_bounds__(AUX_THREADS)
    scatter_kernel(const SysDev* __restrict__ sysv, int sys, int i0, const double* __restrict__ in,
                   Real* __restrict__ fbuf) {
    const SysDev& S = sysv[sys];
    const int64_t site = int64_t(blockIdx.x) * AUX_THREADS + threadIdx.x;
    if (site >= S.n_sites) return;
    const int i = i0 + blockIdx.y;
    fbuf[pulled_element<L>(S, int(site), i)] =
        Real(in[int64_t(blockIdx.y) * S.n_sites + site] - (i == 0 ? S.rho_c : 0.0));
}

// Sums of the pulled populations of a site, rv = sum_i f_i, mv = sum_i c_i f_i, by
// integer additions: the per-population work and the conversions stay off the FP64
// units, which do two operations per clock and SM.  FP32 fields to 2^-57 of the
// largest population (FixedSum; compensated FP32 sums with eight conversions per
// site took 57 us for 2^20 sites, now 47), FP64 fields to 2^-116 (WideSum;
// compensated FP64 sums, to 2^-106, took 0.39 ms for 573,440 sites).  Outside
// their range: FP64 sums, compensated (Knuth's TwoSum).
template <class L, class Real>
__device__ __forceinline__ void site_sums(const Real (&f)[L::Q], double& rv, double (&mv)[3]) {
    bool in_range;
    if constexpr (sizeof(Real) == 8) {
        const WideSum<L::Q> s(f);
        __int128 r = 0, m[3] = {0, 0, 0};
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
            const __int128 v = s.add(i);
            r += v;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (L::c(i, a) == 1) m[a] += v;
                if (L::c(i, a) == -1) m[a] -= v;
            }
        }
        rv = s.value(r);
        for (int a = 0; a < 3; ++a) mv[a] = s.value(m[a]);
        in_range = s.in_range();
    } else {
        const FixedSum<Real, L::Q> s(f);
        int64_t r = 0, m[3] = {0, 0, 0};
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
            r += s.m[i];
#pragma unroll
            for (int a = 0; a < 3; ++a) m[a] += L::c(i, a) * s.m[i];
        }
        rv = s.value(r);
        for (int a = 0; a < 3; ++a) mv[a] = s.value(m[a]);
        in_range = s.in_range();
    }
    if (!in_range) {
        double v[4] = {0.0, 0.0, 0.0, 0.0}, c[4] = {0.0, 0.0, 0.0, 0.0};
        auto add = [&](int k, double x) {
            const double t = v[k] + x, y = t - v[k];
            c[k] += (v[k] - (t - y)) + (x - y);
            v[k] = t;
        };
        for (int i = 0; i < L::Q; ++i) {
            add(0, double(f[i]));
            for (int a = 0; a < 3; ++a)
                if (L::c(i, a) != 0) add(1 + a, L::c(i, a) * double(f[i]));
        }
        auto sum = [&](int k) { return v[k] - v[k] == 0.0 ? v[k] + c[k] : v[k]; };    // (an overflow has no remainder)
        rv = sum(0);
        for (int a = 0; a < 3; ++a) mv[a] = sum(1 + a);
    }
}

// Observable site pass: d(r) = rho(r, t) - rho_c = sum_i delta f_i(r - c_i) and
// j(r) = sum_i c_i f_i(r - c_i) (site_sums).  Writes d and per-item partial sums (sum d, sum jx,
// sum jy, sum jz) in FP64, and, when jout is not null, the momentum field
// j_a(r) at jout + a * jstride (D components).
template <class L, class Real>
__global__ void __launch_bounds__(AUX_THREADS)
    obs_site_kernel(const SysDev* __restrict__ sysv, const int4* __restrict__ items, const Real* __restrict__ fbuf,
                    double* __restrict__ d, double* __restrict__ partial, double* __restrict__ jout,
                    int64_t jstride) {
    __shared__ BlockSum<4, AUX_THREADS> sh;
    const int4 it = items[blockIdx.x];
    const SysDev& S = sysv[it.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz;
    const Real* fb = fbuf + S.pop_offset;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int j = 0; j < SITES_PER_THREAD; ++j) {
        const int site = it.y + j * AUX_THREADS + threadIdx.x;
        if (site >= it.z) break;
        int x, y, z;
        site_coords(site, nx, ny, x, y, z);
        // offsets of the pulled rows and columns (index 1 + c of the velocity)
        const int X[3] = {wrap1(x + 1, nx), x, wrap1(x - 1, nx)};
        const int Y[3] = {wrap1(y + 1, ny) * nx, y * nx, wrap1(y - 1, ny) * nx};
        const int Z[3] = {L::D == 3 ? wrap1(z + 1, nz) * nx * ny : 0, z * nx * ny,
                          L::D == 3 ? wrap1(z - 1, nz) * nx * ny : 0};
        Real f[L::Q];
#pragma unroll
        for (int i = 0; i < L::Q; ++i)
            f[i] = fb[i * S.ns + X[1 + L::c(i, 0)] + Y[1 + L::c(i, 1)] + Z[1 + L::c(i, 2)]];
        double rv, mv[3];
        site_sums<L, Real>(f, rv, mv);
        d[S.site_offset + site] = rv;
        if (jout) {
#pragma unroll
            for (int a = 0; a < L::D; ++a) jout[a * jstride + S.site_offset + site] = mv[a];
        }
        acc[0] += rv;
        acc[1] += mv[0];
        acc[2] += mv[1];
        if constexpr (L::D == 3) acc[3] += mv[2];
    }
    block_sum(acc, sh);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k) partial[int64_t(blockIdx.x) * 4 + k] = acc[k];
    }
}

}  // namespace lbf

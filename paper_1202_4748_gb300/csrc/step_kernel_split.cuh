// Split form of the fused step: a moment pass writes the density and momentum
// of every site (from the 19 populations pulled to it, once per site), and a
// collision pass reads that field around each block of sites and writes the
// post-collision populations.  With every mode at tau = 1 the collision needs
// nothing else; with other rates it pulls the site's populations again.
//
// Against the z-marching kernels, which re-form the density on the halo of
// every column and walk it plane by plane, this trades 16 extra bytes written
// and about 35 read per site (both from L2 while the ensemble fits there) for
// having no serial chain: every site of every block is in flight at once.  A
// marching CTA takes about 1.6 us per plane however few CTAs there are, so an
// ensemble that gives it less than a CTA per SM waits for latency alone.
#pragma once

#include "collide_d3q19.cuh"
#include "step_kernels.cuh"

namespace lbf {

// Density deviation and momentum of every site of the items: mom[site] = drho,
// mom[(1 + a) stride + site] = j_a, each summed in the order of the fused
// kernels (from 0, direction by direction).  One site per thread (any sides).
template <class L, class Real, int NT>
__global__ void __launch_bounds__(NT)
    moments_kernel(const SysDev* __restrict__ sysv, const int4* __restrict__ items, const Real* __restrict__ fbuf,
                   Real* __restrict__ mom, int64_t stride) {
    const int4 it = items[blockIdx.x];
    const SysDev& S = sysv[it.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz, N = S.ns;
    const Real* __restrict__ fb = fbuf + S.pop_offset;
    Real* __restrict__ out = mom + S.site_offset;
    grid_wait();
    for (int site = it.y + int(threadIdx.x); site < it.z; site += NT) {
        const int r = site / nx, x = site - r * nx, z = r / ny, y = r - z * ny;
        const Nbr nb(x, y, z, nx, ny, nz, L::D == 3);
        Real f[L::Q], j[3];
        pull_site<L, Real>(fb, N, nb, f);
        Real v = Real(0);
        sfor<0, L::Q>([&](auto I) { v = vadd(v, f[decltype(I)::value]); });
        momentum_of<L, Real>(f, j);
        out[site] = v;
        sfor<0, L::D>([&](auto C) { out[(1 + int(C)) * stride + site] = j[decltype(C)::value]; });
    }
    grid_release();
}

// The same with four x-adjacent sites per thread (FP32, every nx a multiple of
// 4): one aligned 16-byte load per population, the value that the c_x = +-1
// directions pull across the quad's edge from the neighbouring lane, or loaded
// where that lane holds another row's quad or none.  A site costs 70
// instructions instead of 255, and a warp has 9.7 KB of loads in flight.
template <class L, int NT>
__global__ void __launch_bounds__(NT)
    moments_quad_kernel(const SysDev* __restrict__ sysv, const int4* __restrict__ items,
                        const float* __restrict__ fbuf, float* __restrict__ mom, int64_t stride) {
    const int4 it = items[blockIdx.x];
    const SysDev& S = sysv[it.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz, N = S.ns;
    const float* __restrict__ fb = fbuf + S.pop_offset;
    float* __restrict__ out = mom + S.site_offset;
    const int lane = threadIdx.x & 31;
    grid_wait();
    // every lane of a warp runs the same iterations (the shuffles need all of
    // them); a lane past the end repeats the item's last quad and stores nothing
    for (int s0 = it.y + 4 * int(threadIdx.x - lane); s0 < it.z; s0 += 4 * NT) {
        const bool mine = s0 + 4 * lane < it.z;
        const int site = mine ? s0 + 4 * lane : it.z - 4;
        const int r = site / nx, x = site - r * nx, z = r / ny, y = r - z * ny;
        const Nbr nb(x, y, z, nx, ny, nz, L::D == 3);
        const bool left = x == 0 || lane == 0, right = x + 4 == nx || lane == 31 || !mine || s0 + 4 * lane + 4 >= it.z;
        const int xl = x == 0 ? nx - 1 : x - 1, xr = x + 4 == nx ? 0 : x + 4;
        float4 g[L::Q];
        float e[L::Q];
        sfor<0, L::Q>([&](auto I) {
            constexpr int i = I;
            constexpr int cx = L::c(i, 0);
            const float* row = fb + (i * N + nb.Y[1 - L::c(i, 1)] + nb.Z[1 - L::c(i, 2)]);
            g[i] = *reinterpret_cast<const float4*>(row + x);
            if constexpr (cx == 1) e[i] = left ? row[xl] : 0.0f;
            if constexpr (cx == -1) e[i] = right ? row[xr] : 0.0f;
        });
        float2 v01 = make_float2(0.0f, 0.0f), v23 = v01;
        float2 j01[3] = {v01, v01, v01}, j23[3] = {v01, v01, v01};
        sfor<0, L::Q>([&](auto I) {
            constexpr int i = I;
            constexpr int cx = L::c(i, 0);
            const float4 w = g[i];
            float2 a01, a23;
            if constexpr (cx == 0) {
                a01 = make_float2(w.x, w.y);
                a23 = make_float2(w.z, w.w);
            } else if constexpr (cx == 1) {
                const float p = __shfl_up_sync(0xffffffffu, w.w, 1);
                a01 = make_float2(left ? e[i] : p, w.x);
                a23 = make_float2(w.y, w.z);
            } else {
                const float p = __shfl_down_sync(0xffffffffu, w.x, 1);
                a01 = make_float2(w.y, w.z);
                a23 = make_float2(w.w, right ? e[i] : p);
            }
            v01 = vadd(v01, a01);
            v23 = vadd(v23, a23);
            sfor<0, L::D>([&](auto C) {
                constexpr int c = C;
                if constexpr (L::c(i, c) == 1) {
                    j01[c] = vadd(j01[c], a01);
                    j23[c] = vadd(j23[c], a23);
                }
                if constexpr (L::c(i, c) == -1) {
                    j01[c] = vsub(j01[c], a01);
                    j23[c] = vsub(j23[c], a23);
                }
            });
        });
        if (mine) {
            *reinterpret_cast<float4*>(out + site) = make_float4(v01.x, v01.y, v23.x, v23.y);
            sfor<0, L::D>([&](auto C) {
                constexpr int c = C;
                *reinterpret_cast<float4*>(out + (1 + c) * stride + site) =
                    make_float4(j01[c].x, j01[c].y, j23[c].x, j23[c].y);
            });
        }
    }
    grid_release();
}

// Two sites stacked in z per thread (paired FP32): at<cx, cy, cz>() is the pair
// of values at (x + cx, y + cy, z + cz) and one plane above, from the four
// planes z - 1 .. z + 2 of row pitch PX.
template <int PX>
struct ZPlanes {
    const float *m, *o, *p, *q;
    int c;
    template <int CX, int CY, int CZ>
    __device__ __forceinline__ float2 at() const {
        constexpr int off = CX + PX * CY;
        if constexpr (CZ == -1) return make_float2(m[c + off], o[c + off]);
        else if constexpr (CZ == 0) return make_float2(o[c + off], p[c + off]);
        else return make_float2(p[c + off], q[c + off]);
    }
};

// Collision pass (D3Q19, FP32, every mode at tau = 1): a CTA owns a TX x TY
// column and walks a chunk of A.zc planes, two planes per iteration, one pair
// of sites stacked in z per thread.  Every load and store is then a row of
// consecutive sites, whatever the parity of the sides.  Density planes come
// from the moment field by 4-byte cp.async into a ring, two iterations before
// the Laplacian that needs them; the Laplacian (Guo form) of planes z + 3,
// z + 4 and the collision of planes z, z + 1 share one phase, so there is one
// CTA barrier per iteration; the momenta of the next pair are in flight across
// it.  Rings of 8 planes: the collision of z reads density z, z + 1 (z - 1 ..
// z + 2 for the modified equilibrium) and Laplacian z - 1 .. z + 2, the
// Laplacian pass reads density z + 2 .. z + 5 and writes Laplacian z + 3,
// z + 4, the copies write density z + 6, z + 7, and a warp still in the
// iteration before reads nothing below density z - 3 and Laplacian z - 3.
template <int CP, int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX* TY, MINB)
    collide_march_kernel(const StepArgs<float> A, const float* __restrict__ mom, int64_t stride) {
    constexpr int H = CP == GUO ? 2 : 1;
    constexpr int NT = TX * TY, R = 8;
    constexpr int SX = TX + 2 * H, SY = TY + 2 * H, SP = SX * SY;
    constexpr int LX = TX + 2, LY = TY + 2, LP = CP == GUO ? LX * LY : 1;
    constexpr int PPT = (SP + NT - 1) / NT;           // footprint sites per thread
    constexpr int AHEAD = CP == GUO ? 5 : 2;          // highest density plane an iteration reads, minus z
    __shared__ float srho[R * SP];
    __shared__ float slap[R * LP];

    const int4 tl = A.tiles[blockIdx.x];
    const SysDev& S = A.sys[tl.x];
    const SysPhys<float> P = A.phys[tl.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz, N = S.ns, pl = nx * ny;
    const int z0 = tl.w, z1 = min(z0 + A.zc, nz);
    const int tid = threadIdx.x;
    const int lx = tid % TX, ly = tid / TX;
    const int x = tl.y + lx, y = tl.z + ly;
    const bool own = x < nx && y < ny;
    const float* __restrict__ rho_g = mom + S.site_offset;
    float* __restrict__ fo = A.fout + S.pop_offset + (y * nx + x);
    const float* __restrict__ jg = rho_g + stride + (y * nx + x);
    const int64_t js = stride;

    // wrapped in-plane offset of the thread's footprint sites (-1: not needed)
    int foot[PPT];
    sfor<0, PPT>([&](auto K) {
        constexpr int k = K;
        const int i = tid + k * NT, gx = tl.y + i % SX - H, gy = tl.z + i / SX - H;
        foot[k] = i < SP && gx < nx + H && gy < ny + H ? wrapm(gx, nx) + wrapm(gy, ny) * nx : -1;
    });
    auto slot = [](int rel) { return rel & (R - 1); };   // rel = plane - z0 + R
    auto fetch = [&](int zz) {                           // density plane zz into its ring slot
        const float* src = rho_g + wrapm(zz, nz) * pl;
        float* dst = srho + slot(zz - z0 + R) * SP + tid;
        sfor<0, PPT>([&](auto K) {
            constexpr int k = K;
            if (foot[k] >= 0) cp_async4(dst + k * NT, src + foot[k]);
        });
    };
    const int zlast = z1 - 1 + H;                        // last density plane any collision of the chunk needs
    auto laplacian2 = [&](int zl) {                      // Laplacian planes zl, zl + 1
        if constexpr (CP == GUO) {
            const int r = zl - z0 + R;
            const float* pm = srho + slot(r - 1) * SP;
            const float* p0 = srho + slot(r) * SP;
            const float* p1 = srho + slot(r + 1) * SP;
            const float* p2 = srho + slot(r + 2) * SP;
            float* l0 = slap + slot(r) * LP;
            float* l1 = slap + slot(r + 1) * LP;
            for (int i = tid; i < LP; i += NT) {
                const int c = (i / LX + 1) * SX + i % LX + 1;
                const ZPlanes<SX> rv{pm, p0, p1, p2, c};
                const float2 lap = lap_d3q19<float2>(rv);
                l0[i] = lap.x;
                l1[i] = lap.y;
            }
        }
    };
    float2 jn[3];
    auto momenta = [&](int z) {                          // the pair's momenta (the second site may not exist)
        sfor<0, 3>([&](auto C) { jn[decltype(C)::value] = make_float2(0.0f, 0.0f); });
        if (own && z < z1) {
            const int up = z + 1 < z1 ? pl : 0;
            sfor<0, 3>([&](auto C) {
                constexpr int c = C;
                const float* q = jg + c * js + z * pl;
                jn[c] = make_float2(q[0], q[up]);
            });
        }
    };

    grid_wait();
    const NoiseKey key = noise_key(S, *A.step_ptr + A.k);
    for (int zz = z0 - H; zz <= min(z0 + AHEAD - (CP == GUO ? 2 : 0), zlast); ++zz) fetch(zz);
    cp_async_commit();
    if constexpr (CP == GUO) {
        for (int zz = z0 + AHEAD - 1; zz <= min(z0 + AHEAD, zlast); ++zz) fetch(zz);
        cp_async_commit();
    }
    momenta(z0);
    if constexpr (CP == GUO) {
        cp_async_wait<1>();
        __syncthreads();
        laplacian2(z0 - 1);
        laplacian2(z0 + 1);
    }
    for (int z = z0; z < z1; z += 2) {
        float2 jm[3];
        sfor<0, 3>([&](auto C) { jm[decltype(C)::value] = jn[decltype(C)::value]; });
        cp_async_wait<0>();                              // density up to plane z + AHEAD has landed (this thread's copies)
        __syncthreads();
        if (z + 2 < z1) {
            for (int zz = z + AHEAD + 1; zz <= min(z + AHEAD + 2, zlast); ++zz) fetch(zz);
            momenta(z + 2);
        }
        cp_async_commit();
        if (CP == GUO && z + 2 < z1) laplacian2(z + 3);
        if (z + 2 >= z1) grid_release();
        if (own) {
            const bool two = z + 1 < z1;
            const int site = y * nx + x + z * pl;
            const uint2 sites = make_uint2(site, two ? site + pl : site);
            const int r = z - z0 + R;
            const int c = (ly + H) * SX + lx + H;
            const float* d0 = srho + slot(r) * SP + c;
            const float* d1 = srho + slot(two ? r + 1 : r) * SP + c;   // past the chunk the second lane repeats the first
            const float2 drho = make_float2(d0[0], d1[0]);
            float2 f[19];
            if constexpr (CP == GUO) {
                const ZPlanes<LX> lv{slap + slot(r - 1) * LP, slap + slot(r) * LP, slap + slot(r + 1) * LP,
                                     slap + slot(r + 2) * LP, (ly + 1) * LX + lx + 1};
                collide_d3q19_tau1<float2>(f, drho, jm[0], jm[1], jm[2], lv, P, key, sites, A.status);
            } else {
                const ZPlanes<SX> rv{srho + slot(r - 1) * SP, srho + slot(r) * SP, srho + slot(r + 1) * SP,
                                     srho + slot(r + 2) * SP, c};
                collide_d3q19_modeq_tau1<float2>(f, drho, jm[0], jm[1], jm[2], rv, P, key, sites, A.status);
            }
            sfor<0, 19>([&](auto I) { fo[decltype(I)::value * N + z * pl] = f[decltype(I)::value].x; });
            if (two) sfor<0, 19>([&](auto I) { fo[decltype(I)::value * N + (z + 1) * pl] = f[decltype(I)::value].y; });
        }
    }
}

}  // namespace lbf

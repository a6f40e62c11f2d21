// Split form of the fused step: a moment pass writes the density and momentum
// of every site (from the populations pulled to it, once per site), and a
// collision pass reads that field around each column of sites and writes the
// post-collision populations.  In FP32 with every mode at tau = 1 the collision
// needs nothing else; with other rates, or in FP64, it pulls the site's
// populations again and the moment pass writes the density alone (FP64: so that
// the field fits the scratch of a sample, which it shares).
//
// Each kernel is launched before its predecessor has ended and waits for it
// behind its prologue, which reads only what no kernel writes (the plan's
// records).  The buffers that kernels write are not `const __restrict__` here:
// that promises read-only data for the whole kernel, which these are only behind
// the wait.  It lets its successor's CTAs start when it has done its
// work, or, where both fit on an SM each (`early`), as soon as it runs itself:
// 16^3 5.8 -> 5.2 us per step.  With more CTAs those of the successor go to the
// few SMs with room, several to each, and stay there (32^3 6.0 -> 8.2 us).
//
// Against the kernels that form the density on the halo of every column, this
// trades 16 bytes written and about 35 read per FP32 site (from L2 while the
// ensemble fits there) for forming each density once, which is what the FP64
// path needs (its units do two operations per clock and SM), and for short
// chunks: a paired CTA takes 1.53 us per plane however few CTAs there are, so an
// ensemble that gives it less than a CTA per SM waits for latency alone.
#pragma once

#include "collide_d2q9.cuh"
#include "collide_d3q19.cuh"
#include "step_kernels.cuh"

namespace lbf {

// Density deviation and (J) momentum of every site of the items: mom[site] =
// drho, mom[(1 + a) stride + site] = j_a, each summed in the order of the fused
// kernels (from 0, direction by direction).  One site per thread (any sides).
template <class L, class Real, bool J, int NT>
__global__ void __launch_bounds__(NT)
    moments_kernel(const SysDev* __restrict__ sysv, const int4* __restrict__ items, const Real* fbuf,
                   Real* mom, int64_t stride, int early) {
    const int4 it = items[blockIdx.x];
    const SysDev& S = sysv[it.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz, N = S.ns;
    const Real* fb = fbuf + S.pop_offset;
    Real* out = mom + S.site_offset;
    grid_wait();
    if (early) grid_release();
    for (int site = it.y + int(threadIdx.x); site < it.z; site += NT) {
        const int r = site / nx, x = site - r * nx, z = r / ny, y = r - z * ny;
        const Nbr nb(x, y, z, nx, ny, nz, L::D == 3);
        Real f[L::Q];
        pull_site<L, Real>(fb, N, nb, f);
        out[site] = density_of(f);
        if constexpr (J) {
            Real j[3];
            momentum_of<L, Real>(f, j);
            sfor<0, L::D>([&](auto C) { out[(1 + int(C)) * stride + site] = j[decltype(C)::value]; });
        }
    }
    grid_release();
}

// The same with four x-adjacent sites per thread (FP32, every nx a multiple of
// 4): one aligned 16-byte load per population, the value that the c_x = +-1
// directions pull across the quad's edge from the neighbouring lane, or loaded
// where that lane holds another row's quad or none.  A site costs 70
// instructions instead of 255, and a warp has 9.7 KB of loads in flight.
template <class L, bool J, int NT>
__global__ void __launch_bounds__(NT)
    moments_quad_kernel(const SysDev* __restrict__ sysv, const int4* __restrict__ items,
                        const float* fbuf, float* mom, int64_t stride, int early) {
    const int4 it = items[blockIdx.x];
    const SysDev& S = sysv[it.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz, N = S.ns;
    const float* fb = fbuf + S.pop_offset;
    float* out = mom + S.site_offset;
    const int lane = threadIdx.x & 31;
    grid_wait();
    if (early) grid_release();
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
            if constexpr (J) sfor<0, L::D>([&](auto C) {
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
            if constexpr (J) sfor<0, L::D>([&](auto C) {
                constexpr int c = C;
                *reinterpret_cast<float4*>(out + (1 + c) * stride + site) =
                    make_float4(j01[c].x, j01[c].y, j23[c].x, j23[c].y);
            });
        }
    }
    grid_release();
}

// The thread's sites are W = 1 site, or 2 stacked in z (paired FP32):
// at<cx, cy, cz>() is the value (or pair of values) at (x + cx, y + cy, z + cz)
// from the planes z - 1 .. z + W of row pitch PX.
template <class V, int PX>
struct ZPlanes {
    using S = typename VT<V>::S;
    const S* p[2 + VT<V>::W];
    int c;
    template <int CX, int CY, int CZ>
    __device__ __forceinline__ V at() const {
        constexpr int off = CX + PX * CY;
        if constexpr (VT<V>::W == 2) return make_float2(p[1 + CZ][c + off], p[2 + CZ][c + off]);
        else return p[1 + CZ][c + off];
    }
};

// Collision pass of the split step on D3Q19: a CTA owns a TX x TY column and
// walks a chunk of A.zc planes, W per iteration: two with paired FP32, one site
// per lane of the pair, else one.  Every load and store is then a row of
// consecutive sites, whatever the parity of the sides.  Density planes come
// from the moment field by cp.async into a ring, an iteration before the
// Laplacian that needs them; the Laplacian (Guo form) of planes z + W + 1 ..
// z + 2 W and the collision of planes z .. z + W - 1 share one phase, so there
// is one CTA barrier per iteration; the momenta of the next sites are in flight
// across it.  With rates other than 1 (MODE 0 and 1) and in FP64 a thread pulls
// its sites' populations instead, requested before the Laplacian pass.
//
// Rings of 8 planes: iteration z reads density z .. z + 2 W + 1 (z - 1 .. z + W
// for the modified equilibrium) and Laplacian z - 1 .. z + W, writes Laplacian
// up to z + 2 W, and its copies land in density up to z + 3 W + 1 <= z + 7; no
// warp is in an earlier iteration once they are issued, after the barrier.
//
// 16 x 8 columns, 128 threads: the Laplacian's halo costs 1.4, four
// CTAs per SM decouple the phases.  FP32, tau = 1: bound by issue and, below a
// CTA per SM, by the latency of a chunk (0.87 us per plane).  FP64: bound by
// the FP64 units (two operations per clock and SM).
template <int MODE, int CP, class V, int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX* TY, MINB)
    collide_march_kernel(const StepArgs<typename VT<V>::S> A, const typename VT<V>::S* mom,
                         int64_t stride) {
    using Real = typename VT<V>::S;
    using L = D3Q19;
    constexpr int W = VT<V>::W;
    constexpr bool PULL = MODE != 2 || sizeof(Real) == 8;
    constexpr int H = CP == GUO ? 2 : 1;
    constexpr int NT = TX * TY, R = 8;
    constexpr int SX = TX + 2 * H, SY = TY + 2 * H, SP = SX * SY;
    constexpr int LX = TX + 2, LY = TY + 2, LP = CP == GUO ? LX * LY : 1;
    constexpr int PPT = (SP + NT - 1) / NT;              // footprint sites per thread
    constexpr int AHEAD = CP == GUO ? 2 * W + 1 : W;     // highest density plane an iteration reads, minus z
    __shared__ Real srho[R * SP];
    __shared__ Real slap[R * LP];

    const int4 tl = A.tiles[blockIdx.x];
    const SysDev& S = A.sys[tl.x];
    // fully relaxed: the few parameters it takes, in registers before the first wait
    using Phys = typename std::conditional<MODE == 2, const SysPhys<Real>, const SysPhys<Real>&>::type;
    Phys P = A.phys[tl.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz, N = S.ns, pl = nx * ny;
    const int z0 = tl.w, z1 = min(z0 + A.zc, nz);
    const int tid = threadIdx.x;
    const int lx = tid % TX, ly = tid / TX;
    const int x = tl.y + lx, y = tl.z + ly;
    const bool own = x < nx && y < ny;
    const Real* rho_g = mom + S.site_offset;
    const Real* jg = rho_g + stride + (y * nx + x);
    Real* __restrict__ fo = A.fout + S.pop_offset + (y * nx + x);

    // wrapped in-plane offset of the thread's footprint sites (-1: not needed)
    int foot[PPT];
    sfor<0, PPT>([&](auto K) {
        constexpr int k = K;
        const int i = tid + k * NT, gx = tl.y + i % SX - H, gy = tl.z + i / SX - H;
        foot[k] = i < SP && gx < nx + H && gy < ny + H ? wrapm(gx, nx) + wrapm(gy, ny) * nx : -1;
    });
    auto slot = [](int rel) { return rel & (R - 1); };   // rel = plane - z0 + R
    auto fetch = [&](int zz) {                           // density plane zz into its ring slot
        const Real* src = rho_g + wrapm(zz, nz) * pl;
        Real* dst = srho + slot(zz - z0 + R) * SP + tid;
        sfor<0, PPT>([&](auto K) {
            constexpr int k = K;
            if (foot[k] >= 0) cp_async_elem(dst + k * NT, src + foot[k]);
        });
    };
    const int zlast = z1 - 1 + H;                        // last density plane any collision of the chunk needs
    auto laplacian = [&](int zl) {                       // Laplacian planes zl .. zl + W - 1
        if constexpr (CP == GUO) {
            ZPlanes<V, SX> rv;
            sfor<0, 2 + W>([&](auto K) {
                constexpr int k = K;
                rv.p[k] = srho + slot(zl - z0 + R - 1 + k) * SP;
            });
            Real* l0 = slap + slot(zl - z0 + R) * LP;
            Real* l1 = slap + slot(zl - z0 + R + W - 1) * LP;
            for (int i = tid; i < LP; i += NT) {
                rv.c = (i / LX + 1) * SX + i % LX + 1;
                const V lap = lap_d3q19<V>(rv);
                l0[i] = lane(lap, 0);
                if constexpr (W == 2) l1[i] = lane(lap, 1);
            }
        }
    };
    V jn[3];
    auto momenta = [&](int z) {                          // of the sites (x, y, z ..); the second may not exist
        sfor<0, 3>([&](auto C) { jn[decltype(C)::value] = vk<V>(0.0); });
        if (!PULL && own && z < z1) {
            const int up = z + 1 < z1 ? pl : 0;
            sfor<0, 3>([&](auto C) {
                constexpr int c = C;
                const Real* q = jg + c * stride + z * pl;
                set_lane(jn[c], 0, q[0]);
                if constexpr (W == 2) set_lane(jn[c], 1, q[up]);
            });
        }
    };

    grid_wait();
    if (A.early) grid_release();
    const NoiseKey key = noise_key(S, *A.step_ptr + A.k);
    for (int zz = z0 - H; zz <= min(z0 + AHEAD - (CP == GUO ? W : 0), zlast); ++zz) fetch(zz);
    cp_async_commit();
    if constexpr (CP == GUO) {
        for (int zz = z0 + AHEAD - W + 1; zz <= min(z0 + AHEAD, zlast); ++zz) fetch(zz);
        cp_async_commit();
    }
    momenta(z0);
    if constexpr (CP == GUO) {
        cp_async_wait<1>();
        __syncthreads();
        sfor<0, (2 + W) / W>([&](auto K) { laplacian(z0 - 1 + W * int(K)); });   // planes z0 - 1 .. z0 + W
    }
    for (int z = z0; z < z1; z += W) {
        V jm[3];
        sfor<0, 3>([&](auto C) { jm[decltype(C)::value] = jn[decltype(C)::value]; });
        cp_async_wait<0>();                              // density up to plane z + AHEAD has landed (this thread's copies)
        __syncthreads();
        const bool more = z + W < z1, two = z + 1 < z1;
        if (more) {
            for (int zz = z + AHEAD + 1; zz <= min(z + AHEAD + W, zlast); ++zz) fetch(zz);
            momenta(z + W);
        }
        cp_async_commit();
        V f[19];
        if constexpr (PULL) {
            if (own) {
                const Real* fb = A.fin + S.pop_offset;
                const Nbr nb(x, y, z, nx, ny, nz, true);
                const int pu = two && W == 2 ? z + 1 : z;   // past the chunk the second lane repeats the first
                const int zu[3] = {(pu == 0 ? nz - 1 : pu - 1) * pl, pu * pl, (pu == nz - 1 ? 0 : pu + 1) * pl};
                sfor<0, 19>([&](auto I) {
                    constexpr int i = I;
                    const Real* col = fb + (i * N + nb.X[1 - L::c(i, 0)] + nb.Y[1 - L::c(i, 1)]);
                    set_lane(f[i], 0, col[nb.Z[1 - L::c(i, 2)]]);
                    if constexpr (W == 2) set_lane(f[i], 1, col[zu[1 - L::c(i, 2)]]);
                });
            }
        }
        if (more) laplacian(z + W + 1);
        else grid_release();
        if (own) {
            const int site = y * nx + x + z * pl;
            const int r = z - z0 + R;
            const int c = (ly + H) * SX + lx + H;
            typename SiteIdx<V>::type sites;
            V drho;
            set_lane(drho, 0, srho[slot(r) * SP + c]);
            if constexpr (W == 2) {
                sites = make_uint2(site, two ? site + pl : site);
                set_lane(drho, 1, srho[slot(two ? r + 1 : r) * SP + c]);
            } else {
                sites = site;
            }
            if constexpr (PULL && sizeof(Real) == 8) {
                const FixedSum<double, 19> fs(f);                // as density_of
                sfor<0, 3>([&](auto C) {
                    constexpr int cc = C;
                    int64_t s = 0;
                    double d = 0.0;
                    sfor<1, 19>([&](auto I) {
                        constexpr int i = I;
                        if constexpr (L::c(i, cc) == 1) s += fs.m[i];
                        if constexpr (L::c(i, cc) == -1) s -= fs.m[i];
                    });
                    if (!fs.in_range())
                        sfor<1, 19>([&](auto I) { d += double(L::c(decltype(I)::value, cc)) * f[decltype(I)::value]; });
                    jm[cc] = fs.in_range() ? fs.value(s) : d;
                });
            } else if constexpr (PULL) {
                sfor<0, 3>([&](auto C) {
                    constexpr int cc = C;
                    V s = vk<V>(0.0);
                    sfor<1, 19>([&](auto I) {
                        constexpr int i = I;
                        if constexpr (L::c(i, cc) == 1) s = vadd(s, f[i]);
                        if constexpr (L::c(i, cc) == -1) s = vsub(s, f[i]);
                    });
                    jm[cc] = s;
                });
            }
            ZPlanes<V, CP == GUO ? LX : SX> nv;
            nv.c = CP == GUO ? (ly + 1) * LX + lx + 1 : c;
            sfor<0, 2 + W>([&](auto K) {
                constexpr int k = K;
                nv.p[k] = CP == GUO ? slap + slot(r - 1 + k) * LP : srho + slot(r - 1 + k) * SP;
            });
            if constexpr (MODE != 2)
                collide_d3q19_rates<MODE, CP, V>(f, drho, jm[0], jm[1], jm[2], nv, P, key, sites, A.status);
            else if constexpr (CP == GUO)
                collide_d3q19_tau1<V>(f, drho, jm[0], jm[1], jm[2], nv, P, key, sites, A.status);
            else
                collide_d3q19_modeq_tau1<V>(f, drho, jm[0], jm[1], jm[2], nv, P, key, sites, A.status);
            sfor<0, 19>([&](auto I) { fo[decltype(I)::value * N + z * pl] = lane(f[decltype(I)::value], 0); });
            if constexpr (W == 2) {
                if (two)
                    sfor<0, 19>([&](auto I) { fo[decltype(I)::value * N + (z + 1) * pl] = lane(f[decltype(I)::value], 1); });
            }
        }
    }
}

}  // namespace lbf

// Fused step of the modified-equilibrium coupling on D3Q19.
//
// The paper prints its modified equilibrium (Eq. 65) for D2Q9 only.  On D3Q19
// the library uses the same structure with the isotropic weights 3 t_i,
//   f_i^eq = 3 t_i [p0 - kappa rho lap rho + rho c_i.u + (3/2)(c_ia c_ib - delta_ab/3) X_ab]
//          + kappa t_i [(9/2)(c_i.g)^2 - (9/2) c_i^2 |g|^2 + (9/2) |g|^2]      (i >= 1),
//   f_0^eq = rho - sum_{i>=1} f_i^eq,
// g = grad rho, X_ab = rho u_a u_b + nu (u_a g_b + u_b g_a + u.g delta_ab):
// the square-gradient terms are the rotation-invariant form of the printed
// D2Q9 weights with the one coefficient that the second-moment condition
// (Eq. 63) leaves free kept at its D2Q9 value, -9/2 for c_i^2 |g|^2.  Every
// moment condition of Eqs. 62-64 then holds in three dimensions.  The noise is
// the lattice-general form of Eq. 68 (exact at kappa = 0 for this
// equilibrium, whose linearisation is the Landau-pressure one).
//
// The coupling needs the density on the 3 x 3 x 3 neighbourhood only, so the
// z-marching kernel keeps one footprint ring of radius 1.  It runs FP32 with
// every mode at tau = 1 (collide_d3q19_modeq_tau1, the closed form of the
// moments on the D3Q19 basis); the other settings take the split step.
#pragma once

#include "step_kernels.cuh"

namespace lbf {

// z-marching step for the modified equilibrium on D3Q19: a CTA owns a TX x TY
// column and walks a chunk of A.zc planes; iteration zz forms the density of
// footprint plane zz (tile + 1 site, from the pulled populations) and the
// momentum of the tile sites, so that the collision needs no second pull, into a ring of 4 planes, and after one barrier collides plane
// zz - 1, whose density neighbourhood (planes zz - 2 .. zz) is complete.  The
// next iteration writes the slot of plane zz - 3, which no collision of
// iteration zz reads, and no thread starts it before every thread has passed
// the barrier of iteration zz.
template <class L, int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX* TY, MINB) step_kernel_zm(const StepArgs<float> A) {
    using Real = float;
    static_assert(L::D == 3, "z-marching is for 3-D lattices");
    constexpr int Q = L::Q;
    constexpr int SX = TX + 2, SY = TY + 2, SP = SX * SY, NT = TX * TY, NR = 4;
    __shared__ Real srho[NR * SP];
    __shared__ Real sj[NR * 3 * NT];

    const int4 tl = A.tiles[blockIdx.x];
    const SysDev& S = A.sys[tl.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz;
    const int N = S.ns;
    const Real* __restrict__ fb = A.fin + S.pop_offset;
    Real* __restrict__ fo = A.fout + S.pop_offset;
    const int z0 = tl.w, z1 = min(z0 + A.zc, nz);
    const int64_t step = *A.step_ptr + A.k;
    const int tid = threadIdx.x;
    const int tx = tid % TX, ty = tid / TX;
    const int x = tl.y + tx, y = tl.z + ty;
    const bool valid_xy = x < nx && y < ny;
    const bool sm = S.small != 0;

    for (int zz = z0 - 1; zz <= z1; ++zz) {
        const int slot = (zz - z0 + 1) & (NR - 1);
        for (int idx = tid; idx < SP; idx += NT) {
            const int px = idx % SX, py = idx / SX;
            const int gx = tl.y + px - 1, gy = tl.z + py - 1;
            Real v = Real(0);
            if (gx < nx + 1 && gy < ny + 1) {
                const Nbr nb(sm ? wrapm(gx, nx) : wrap2(gx, nx), sm ? wrapm(gy, ny) : wrap2(gy, ny),
                             sm ? wrapm(zz, nz) : wrap2(zz, nz), nx, ny, nz, true);
                Real g[Q];
                pull_site<L, Real>(fb, N, nb, g);
                sfor<0, Q>([&](auto I) { v += g[decltype(I)::value]; });
                if (px >= 1 && px <= TX && py >= 1 && py <= TY) {
                    Real jm[3];
                    momentum_of<L, Real>(g, jm);
                    sfor<0, 3>([&](auto C) {
                        sj[(slot * 3 + int(C)) * NT + (py - 1) * TX + (px - 1)] = jm[decltype(C)::value];
                    });
                }
            }
            srho[slot * SP + idx] = v;
        }
        __syncthreads();
        const int zc = zz - 1;
        if (zc >= z0 && valid_xy) {
            const int cs = (zc - z0 + 1) & (NR - 1), rm = (zc - z0) & (NR - 1), rp = (zc - z0 + 2) & (NR - 1);
            const int c = (ty + 1) * SX + (tx + 1);
            const RingView<Real, SX> rv{srho, rm * SP, cs * SP, rp * SP, c};
            const Real drho = srho[cs * SP + c];
            Real f[Q];
            Real jc[3];
            sfor<0, 3>([&](auto C) { jc[decltype(C)::value] = sj[(cs * 3 + int(C)) * NT + tid]; });
            const int site = site_index(x, y, zc, nx, ny);
            collide_d3q19_modeq_tau1<Real>(f, drho, jc[0], jc[1], jc[2], rv, A.phys[tl.x], noise_key(S, step),
                                           uint32_t(site), A.status);
            sfor<0, Q>([&](auto I) {
                constexpr int i = I;
                fo[i * N + site] = f[i];
            });
        }
    }
}

}  // namespace lbf

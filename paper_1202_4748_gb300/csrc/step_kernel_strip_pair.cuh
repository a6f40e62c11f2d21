// Row-marching strips of the D2Q9 modified-equilibrium step with two sites
// per lane (FP32, every mode at tau = 1).
//
// A warp owns 64 consecutive sites of a row (tile (system, x0, y0), x0 a
// multiple of 64) and walks A.zc rows; lane l holds the sites x0 + 2l and
// x0 + 2l + 1 as one float2.  The 9 populations of a footprint row, each from the
// row that it is pulled from, columns x0 - 4 .. x0 + 67, are copied into shared
// memory by 162 copies of 16 bytes, issued a row ahead; the populations stand
// there by c_y, so that the copies of one source row differ between lanes by a
// constant.  A lane then reads its shifted pairs (the pull's -c_x), forms the
// density of both sites, gets the neighbours' densities by shuffles (lanes 0 and
// 31 sum those of the sites x0 - 1 and x0 + 64), and three density rows stay in
// registers.  With every mode at tau = 1 the post-collision state depends on
// the pre-collision populations only through the density and momentum, so the
// site of row yy - 1 collides from the (drho, j) carried over from the
// previous iteration, two sites at once in paired FP32 (the collision of
// collide_d2q9.cuh), and stores an aligned pair per population.
//
// Bound by issue (62 %, the FMA pipe that takes the 64-bit products of the
// generator and the addresses 65 %): 13.7 M sites in 160 systems take 194 us, 0.75
// of the measured copy rate.  Before, with four warps per CTA and the next row's
// loads in registers (168 of them, 12 warps per SM): 224 us; one warp per CTA, so
// that the system's records need no register per lane: 208; an 8-byte copy per
// lane, population and row: 209, of two rows ahead 217 (the copies' addresses
// were a tenth of the instructions); 24 warps per SM 212.
//
// Every x side is a multiple of 4 (checked on the host), so each quad is
// 16-byte aligned and lies inside one row; lanes past the system's last column
// hold the periodic image of their columns for their neighbours and do not
// collide.  The results are bit-identical to the one-site kernels.
#pragma once

#include "collide_d2q9.cuh"
#include "step_kernels.cuh"

namespace lbf {

// Density deviations of one row around a lane's two sites: l = site x - 1,
// c = (x, x + 1), r = site x + 2.
struct PairRow {
    float l;
    float2 c;
    float r;
};

// 3 x 3 density neighbourhood of the two sites: at<cx, cy, 0>() is the pair
// of densities at (x + cx, y + cy) and (x + 1 + cx, y + cy).
struct PairNbr {
    PairRow m, o, p;    // rows y - 1, y, y + 1
    template <int CX>
    __device__ __forceinline__ static float2 pick(const PairRow& w) {
        if constexpr (CX == -1) return make_float2(w.l, w.c.x);
        else if constexpr (CX == 0) return w.c;
        else return make_float2(w.c.y, w.r);
    }
    template <int CX, int CY, int CZ>
    __device__ __forceinline__ float2 at() const {
        if constexpr (CY == -1) return pick<CX>(m);
        else if constexpr (CY == 0) return pick<CX>(o);
        else return pick<CX>(p);
    }
};

// Populations in the staged row, by c_y = -1, 0, 1, and the place of each.
__device__ constexpr int kStripOrder[9] = {4, 6, 7, 0, 1, 2, 3, 5, 8};
constexpr int strip_slot(int i) {
    constexpr int at[9] = {3, 4, 5, 6, 0, 7, 1, 2, 8};
    return at[i];
}

template <int MINB>
__global__ void __launch_bounds__(32, MINB) step_kernel_strip_pair(const StepArgs<float> A) {
    using L = D2Q9;
    constexpr int SW = 72, NQ = SW / 4;              // staged columns x0 - 4 .. x0 + 67
    __shared__ __align__(16) float stage[9 * SW];
    const int lane = threadIdx.x;
    const int4 tl = A.tiles[blockIdx.x];
    // register copies of the per-system records: read once, not again after every row's stores
    const SysDev S = A.sys[tl.x];
    const SysPhys<float> P = A.phys[tl.x];
    const int nx = S.nx, ny = S.ny, N = S.ns;
    const bool sm = S.small != 0;
    const float* __restrict__ fb = A.fin + S.pop_offset;
    float* __restrict__ fo = A.fout + S.pop_offset;
    const int x = tl.y + 2 * lane;
    const bool own = x < nx;
    const bool edge = lane == 0 || lane == 31, left = lane == 0;
    const NoiseKey key = noise_key(S, *A.step_ptr + A.k);
    const int y0 = tl.z, y1 = min(y0 + A.zc, ny);
    // the staged row: populations by c_y (group g: c_y = g - 1, all pulled from
    // one row), 3 x 18 quads each; the lane copies quads lane and lane + 32 of each
    const float* const mine = stage + 4 + 2 * lane;     // column x of the first population
    int from[3][2];
    sfor<0, 6>([&](auto K) {
        constexpr int g = K / 2, k = K % 2;
        const int idx = lane + 32 * k, r = idx / NQ, q = idx - r * NQ;
        const int i = r == 0 ? kStripOrder[3 * g] : (r == 1 ? kStripOrder[3 * g + 1] : kStripOrder[3 * g + 2]);
        from[g][k] = i * N + wrapm(tl.y - 4 + 4 * q, nx);
    });
    auto load_row = [&](int yy) {
        sfor<0, 3>([&](auto G) {
            constexpr int g = G;
            const int src = yy + 1 - g;              // yy - c_y
            const int ro = (sm ? wrapm(src, ny) : wrap2(src, ny)) * nx;
            cp_async16(stage + g * (3 * SW) + 4 * lane, fb + (from[g][0] + ro));
            if (lane + 32 < 3 * NQ) cp_async16(stage + g * (3 * SW) + 4 * lane + 128, fb + (from[g][1] + ro));
        });
        cp_async_commit();
    };
    load_row(y0 - 1);

    float2 pr = make_float2(0.f, 0.f), pjx = pr, pjy = pr;        // (drho, j) of row yy - 1
    PairRow Rm{0.f, pr, 0.f}, R0 = Rm, Rp = Rm;                  // density rows yy - 2, yy - 1, yy
    for (int yy = y0 - 1; yy <= y1; ++yy) {
        cp_async_wait_all();
        __syncwarp();
        // the pull's x shift: f_i(x) = s_i(x - c_x)
        float2 g[9];
        sfor<0, 9>([&](auto I) {
            constexpr int i = I;
            constexpr int cx = L::c(i, 0);
            const float* q = mine + strip_slot(i) * SW;
            if constexpr (cx == 0) g[i] = *reinterpret_cast<const float2*>(q);
            else g[i] = make_float2(q[-cx], q[1 - cx]);
        });
        // edge lanes: the density of the halo site (x0 - 1 or x0 + 64), summed
        // in population order.  (All of a strip's halo densities before its first
        // row, a lane per site, is 4 % fewer instructions and 13 % slower: the
        // scattered reads run rows ahead of the strips that stream the same lines.)
        float rh = 0.f;
        if (edge) {
            sfor<0, 9>([&](auto I) {
                constexpr int i = I;
                rh = vadd(rh, mine[strip_slot(i) * SW - L::c(i, 0) + (left ? -1 : 2)]);
            });
        }
        __syncwarp();
        if (yy < y1) load_row(yy + 1);
        float2 r, jx, jy;
        moments_d2q9<float2>(g, r, jx, jy);
        float rl = __shfl_up_sync(0xffffffffu, r.y, 1);
        float rr = __shfl_down_sync(0xffffffffu, r.x, 1);
        if (lane == 0) rl = rh;
        if (lane == 31) rr = rh;
        Rm = R0;
        R0 = Rp;
        Rp = PairRow{rl, r, rr};
        if (yy > y0 && own) {
            const int y = yy - 1;
            const PairNbr nb{Rm, R0, Rp};
            const uint32_t site = uint32_t(y * nx + x);
            float2 f[9];
            collide_d2q9_modeq<2, float2>(f, pr, pjx, pjy, nb, P, key, make_uint2(site, site + 1u), A.status);
            sfor<0, 9>([&](auto I) {
                constexpr int i = I;
                *reinterpret_cast<float2*>(fo + i * N + site) = f[i];
            });
        }
        pr = r;
        pjx = jx;
        pjy = jy;
    }
}

}  // namespace lbf

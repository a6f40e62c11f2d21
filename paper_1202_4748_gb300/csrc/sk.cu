// Structure factor C(k) = N^-1 |sum_r phi(r) exp(-i k.r)|^2 (Eq. 80), accumulated
// in FP64 over samples for every k of every system.  The discrete Fourier
// transform is taken one axis at a time (x: real -> complex, then y, z) with
// per-side twiddle tables W_n^j = exp(-2 pi i j / n).  Sides up to
// kSkFftMaxElems are transformed by a mixed-radix Stockham FFT, one CTA per
// group of lines in shared memory; longer sides sum each output element's line
// directly in a fixed order.  Shell binning (j(j-1) < |n|^2 <= j(j+1)) happens
// only when the accumulated spectrum is read.
//
// GB300's FP64 units do two operations per clock and SM, so the transforms are
// bound by their arithmetic, and what is left out counts: the fields are real,
// so the x pass of an even side is a complex FFT of half the length, only the
// kx <= S/2 half of the spectrum is carried through the other axes, and the
// last pass adds both of a mode's squared moduli (k and -k) to the accumulated
// spectra.  All fields of a sample (order parameter, momentum components) go
// through each pass in one launch: 3 launches on D3Q19 instead of 15.
#include "lattice_kernels.cuh"
#include "lb_launch.h"

namespace lbf {

namespace {

__global__ void sk_twiddle_kernel(double* __restrict__ tw, const int* __restrict__ sides,
                                  const int* __restrict__ offs, int n_tables, int max_n) {
    const int t = blockIdx.y;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_tables) return;
    const int n = sides[t];
    if (j >= n || j >= max_n) return;
    double s, c;
    sincospi(-2.0 * double(j) / double(n), &s, &c);
    tw[2 * (offs[t] + j)] = c;
    tw[2 * (offs[t] + j) + 1] = s;
}

// item: (system, first element, end element, unused); element e of a system
// enumerates its sites in [z][y][x] order, and names the output (k_x, y, z) etc.
// With dbar the input is phi = (d - dbar) / (rho_c + dbar); without (null) it
// is the field d itself.
__global__ void __launch_bounds__(AUX_THREADS)
    sk_x_kernel(const SkSys* __restrict__ skv, const int4* __restrict__ items,
                const double* __restrict__ d, const double* __restrict__ dbar, const double* __restrict__ tw,
                double* __restrict__ out) {
    const int4 it = items[blockIdx.x];
    const SkSys K = skv[it.x];
    const double db = dbar ? dbar[2 * it.x] : 0.0;
    const double inv_rbar = dbar ? dbar[2 * it.x + 1] : 1.0;
    for (int j = 0; j < SITES_PER_THREAD; ++j) {
        const int e = it.y + j * AUX_THREADS + threadIdx.x;
        if (e >= it.z) break;
        const int kx = e % K.nx;
        const int line = e - kx;
        const double* row = d + K.site_offset + line;
        double re = 0.0, im = 0.0;
        int idx = 0;                      // (kx * x) mod nx, advanced incrementally
        for (int x = 0; x < K.nx; ++x) {
            const double phi = (row[x] - db) * inv_rbar;
            re += phi * tw[2 * (K.tw_x + idx)];
            im += phi * tw[2 * (K.tw_x + idx) + 1];
            idx += kx;
            if (idx >= K.nx) idx -= K.nx;
        }
        out[2 * (K.site_offset + e)] = re;
        out[2 * (K.site_offset + e) + 1] = im;
    }
}

__global__ void __launch_bounds__(AUX_THREADS)
    sk_pass_kernel(const SkSys* __restrict__ skv, const int4* __restrict__ items, int axis,
                   const double* __restrict__ tw, const double* __restrict__ in, double* __restrict__ out) {
    const int4 it = items[blockIdx.x];
    const SkSys K = skv[it.x];
    const int n = axis == 1 ? K.ny : K.nz;
    const int64_t stride = axis == 1 ? K.nx : int64_t(K.nx) * K.ny;
    const int toff = axis == 1 ? K.tw_y : K.tw_z;
    for (int j = 0; j < SITES_PER_THREAD; ++j) {
        const int e = it.y + j * AUX_THREADS + threadIdx.x;
        if (e >= it.z) break;
        const int k = int((e / stride) % n);           // output wavenumber index along the axis
        const int64_t base = e - int64_t(k) * stride;  // element with axis coordinate 0
        const double* src = in + 2 * (K.site_offset + base);
        double re = 0.0, im = 0.0;
        int idx = 0;
        for (int y = 0; y < n; ++y) {
            const double ar = src[2 * (int64_t(y) * stride)], ai = src[2 * (int64_t(y) * stride) + 1];
            const double wr = tw[2 * (toff + idx)], wi = tw[2 * (toff + idx) + 1];
            re += ar * wr - ai * wi;
            im += ar * wi + ai * wr;
            idx += k;
            if (idx >= n) idx -= n;
        }
        out[2 * (K.site_offset + e)] = re;
        out[2 * (K.site_offset + e) + 1] = im;
    }
}

__global__ void __launch_bounds__(AUX_THREADS)
    sk_accum_kernel(const SkSys* __restrict__ skv, const int4* __restrict__ items, const double* __restrict__ F,
                    double* __restrict__ acc) {
    const int4 it = items[blockIdx.x];
    const SkSys K = skv[it.x];
    for (int j = 0; j < SITES_PER_THREAD; ++j) {
        const int e = it.y + j * AUX_THREADS + threadIdx.x;
        if (e >= it.z) break;
        const int64_t g = K.site_offset + e;
        const double re = F[2 * g], im = F[2 * g + 1];
        acc[g] += (re * re + im * im) * K.inv_n;
    }
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
// -i a
__device__ __forceinline__ double2 cmi(double2 a) { return make_double2(a.y, -a.x); }

// Complex FFTs of nl lines of length n in shared memory (line l at A + l n),
// with B as the other buffer; returns the one that holds the result.  tw is
// the table of W_S^j, S = n * mul.  Stockham autosort: the stage with radix R
// after sub-transforms of length Ns takes, for butterfly j of a line, the R
// inputs a[j + r n/R] times W_n^(k r n/(Ns R)), k = j mod Ns, and writes their
// R-point DFT to b[(j / Ns) Ns R + k + s Ns]; after the last stage the line is
// in natural order.  Radices 4, 2 and 3, then the odd primes left, whose
// outputs are summed one per thread.
__device__ __forceinline__ double2* fft_lines(double2* A, double2* B, int nl, int n, int mul,
                                              const double2* __restrict__ tw) {
    int Ns = 1;
    for (int m = n; m > 1;) {
        int R = (m % 4 == 0) ? 4 : ((m % 2 == 0) ? 2 : 3);
        while (m % R) R += 2;
        m /= R;
        const int nb = n / R, tstep = mul * (n / (Ns * R));
        if (R > 4) {
            const int S = n * mul, sstep = S / R;
            for (int b = threadIdx.x; b < nl * n; b += blockDim.x) {
                const int l = b / n, o = b - l * n, s = o / nb, j = o - s * nb, k = j % Ns;
                const double2* src = A + l * n + j;
                const int e = k * tstep + s * sstep;          // exponent per input, < 2 S
                double2 v = src[0];
                int idx = 0;
                for (int r = 1; r < R; ++r) {
                    idx += e;
                    while (idx >= S) idx -= S;
                    const double2 w = tw[idx], a = src[r * nb];
                    v.x += a.x * w.x - a.y * w.y;
                    v.y += a.x * w.y + a.y * w.x;
                }
                B[l * n + (j / Ns) * Ns * R + k + s * Ns] = v;
            }
        } else {
            for (int b = threadIdx.x; b < nl * nb; b += blockDim.x) {
                const int l = b / nb, j = b - l * nb, k = j % Ns;
                const double2* src = A + l * n;
                double2* dst = B + l * n + (j / Ns) * Ns * R + k;
                double2 v[4];
                v[0] = src[j];
                if (Ns == 1) {
                    for (int r = 1; r < R; ++r) v[r] = src[j + r * nb];
                } else {
                    for (int r = 1; r < R; ++r) v[r] = cmul(src[j + r * nb], tw[k * r * tstep]);
                }
                if (R == 4) {
                    const double2 s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
                    const double2 s13 = cadd(v[1], v[3]), d13 = cmi(csub(v[1], v[3]));
                    dst[0] = cadd(s02, s13);
                    dst[Ns] = cadd(d02, d13);
                    dst[2 * Ns] = csub(s02, s13);
                    dst[3 * Ns] = csub(d02, d13);
                } else if (R == 2) {
                    dst[0] = cadd(v[0], v[1]);
                    dst[Ns] = csub(v[0], v[1]);
                } else {
                    // w = exp(-2 pi i / 3): X1,2 = v0 - (v1 + v2)/2 -+ i (sqrt(3)/2)(v1 - v2)
                    const double2 t1 = cadd(v[1], v[2]), t2 = csub(v[1], v[2]);
                    const double2 m0 = make_double2(v[0].x - 0.5 * t1.x, v[0].y - 0.5 * t1.y);
                    const double h = 0.86602540378443864676;
                    const double2 rt = make_double2(h * t2.y, -h * t2.x);      // -i (sqrt(3)/2) t2
                    dst[0] = cadd(v[0], t1);
                    dst[Ns] = cadd(m0, rt);
                    dst[2 * Ns] = csub(m0, rt);
                }
            }
        }
        __syncthreads();
        double2* tmp = A;
        A = B;
        B = tmp;
        Ns *= R;
    }
    return A;
}

// x pass: item = (system, first line, line count, field); line l of a system
// is row l in [z][y] order.  Field 0 is phi = (d - dbar)/(rho_c + dbar), field
// f > 0 the momentum component j_(f-1).  Writes the half spectrum kx = 0 .. S/2
// of each line, rows of hx = S/2 + 1 values.  An even side S packs its samples
// as z_j = a_2j + i a_(2j+1), j < S/2 = h: with Z the transform of z,
// F(k) = E + W_S^k O, E = (Z_k + conj Z_(h-k))/2, O = -i (Z_k - conj Z_(h-k))/2.
__global__ void __launch_bounds__(FFT_THREADS)
    fft_x_kernel(const SkSys* __restrict__ skv, const int4* __restrict__ items,
                 const double* __restrict__ d, const double* __restrict__ dbar, const double* __restrict__ jf,
                 int64_t jstride, const double2* __restrict__ twv, double2* __restrict__ F, int64_t fstride) {
    extern __shared__ double2 fft_buf[];
    const int4 it = items[blockIdx.x];
    const SkSys K = skv[it.x];
    const int S = K.nx, hx = S / 2 + 1, nl = it.z;
    const double2* tw = twv + K.tw_x;
    const bool even = S % 2 == 0;
    const int n = even ? S / 2 : S;
    double db = 0.0, inv = 1.0;
    const double* src = it.w == 0 ? d : jf + (it.w - 1) * jstride;
    if (it.w == 0) {
        db = dbar[2 * it.x];
        inv = dbar[2 * it.x + 1];
    }
    src += K.site_offset + int64_t(it.y) * S;
    // the samples in order: interleaved they are the packed complex line
    if (even) {
        double* a = reinterpret_cast<double*>(fft_buf);
        for (int i = threadIdx.x; i < nl * S; i += FFT_THREADS) a[i] = it.w == 0 ? (src[i] - db) * inv : src[i];
    } else {
        for (int i = threadIdx.x; i < nl * S; i += FFT_THREADS)
            fft_buf[i] = make_double2(it.w == 0 ? (src[i] - db) * inv : src[i], 0.0);
    }
    __syncthreads();
    const double2* Z = fft_lines(fft_buf, fft_buf + nl * n, nl, n, even ? 2 : 1, tw);
    double2* out = F + it.w * fstride + K.half_offset + int64_t(it.y) * hx;
    for (int i = threadIdx.x; i < nl * hx; i += FFT_THREADS) {
        const int l = i / hx, k = i - l * hx;
        const double2* z = Z + l * n;
        if (even) {
            const double2 p = z[k == n ? 0 : k], q = z[k == 0 ? 0 : n - k];
            const double2 e = make_double2(0.5 * (p.x + q.x), 0.5 * (p.y - q.y));
            const double2 o = make_double2(0.5 * (p.y + q.y), -0.5 * (p.x - q.x));
            const double2 w = k == 0 ? make_double2(1.0, 0.0) : (k == n ? make_double2(-1.0, 0.0) : tw[k]);
            out[i] = cadd(e, cmul(w, o));
        } else {
            out[i] = z[k];
        }
    }
}

// y pass of a 3-D system, in place on the half spectrum: item = (system, first
// line, line count, field); line l is kx + hx z.
__global__ void __launch_bounds__(FFT_THREADS)
    fft_y_kernel(const SkSys* __restrict__ skv, const int4* __restrict__ items, const double2* __restrict__ twv,
                 double2* __restrict__ F, int64_t fstride) {
    extern __shared__ double2 fft_buf[];
    const int4 it = items[blockIdx.x];
    const SkSys K = skv[it.x];
    const int S = K.ny, hx = K.nx / 2 + 1, nl = it.z;
    double2* f = F + it.w * fstride + K.half_offset;
    // consecutive lines are consecutive kx: a warp reads rows of lines
    auto elem = [&](int i, int& l, int& t) -> int64_t {
        t = i / nl;
        l = i - t * nl;
        const int g = it.y + l, z = g / hx, kx = g - z * hx;
        return kx + int64_t(hx) * (t + int64_t(S) * z);
    };
    for (int i = threadIdx.x; i < nl * S; i += FFT_THREADS) {
        int l, t;
        const int64_t e = elem(i, l, t);
        fft_buf[l * S + t] = f[e];
    }
    __syncthreads();
    const double2* Z = fft_lines(fft_buf, fft_buf + nl * S, nl, S, 1, twv + K.tw_y);
    for (int i = threadIdx.x; i < nl * S; i += FFT_THREADS) {
        int l, t;
        const int64_t e = elem(i, l, t);
        f[e] = Z[l * S + t];
    }
}

__device__ __forceinline__ int wrapk(int k, int n) { return 2 * k < n ? k : k - n; }

// What the spectra of one mode add: |J_x|^2, |n . J|^2 / |n|^2 and the
// transverse rest per component, all over N (0 for the projections at n = 0).
struct ModeSpectra {
    double x, lon, tra;
};
__device__ __forceinline__ ModeSpectra mode_spectra(double a, double b, double c, double2 X, double2 Y, double2 Z,
                                                    int dims, double inv_n) {
    ModeSpectra m{0.0, 0.0, 0.0};
    const double jx2 = X.x * X.x + X.y * X.y;
    m.x = jx2 * inv_n;
    const double nn2 = a * a + b * b + c * c;
    if (nn2 > 0.0) {
        const double pr = a * X.x + b * Y.x + c * Z.x, pi = a * X.y + b * Y.y + c * Z.y;
        const double p2 = (pr * pr + pi * pi) / nn2;
        const double tot = jx2 + Y.x * Y.x + Y.y * Y.y + Z.x * Z.x + Z.y * Z.y;
        m.lon = p2 * inv_n;
        m.tra = (tot - p2) * (dims == 3 ? 0.5 * inv_n : inv_n);
    }
    return m;
}

// Last pass (y in 2-D, z in 3-D) and accumulation: item = (system, first line,
// line count, -); line l is l = kx + hx ky (3-D) or kx.  All nf fields of a
// line are in the CTA, so every mode's spectra are formed where its transforms
// end: acc[k] += |phi(k)|^2 / N, and with momentum components (nf > 1)
// jacc + c stride as ModeSpectra.  A mode with 0 < kx < S/2 stands for -k too:
// its moduli are the same, and so are the projections unless a wrapped
// component is -S/2, whose sign does not flip (n is formed again for it).
__global__ void __launch_bounds__(FFT_THREADS)
    fft_last_kernel(const SkSys* __restrict__ skv, const int4* __restrict__ items, int nf,
                    const double2* __restrict__ twv, const double2* __restrict__ F, int64_t fstride,
                    double* __restrict__ acc, double* __restrict__ jacc, int64_t jstride, int dims) {
    extern __shared__ double2 fft_buf[];
    const int4 it = items[blockIdx.x];
    const SkSys K = skv[it.x];
    const int S = K.nx, hx = S / 2 + 1, nl = it.z;
    const int64_t tstride = dims == 3 ? int64_t(hx) * S : hx;     // along the transformed axis
    const double2* f = F + K.half_offset + it.y;
    for (int i = threadIdx.x; i < nf * nl * S; i += FFT_THREADS) {
        const int fl = i / (nl * S), r = i - fl * (nl * S), t = r / nl, l = r - t * nl;
        fft_buf[(fl * nl + l) * S + t] = f[fl * fstride + l + tstride * t];
    }
    __syncthreads();
    const double2* Z = fft_lines(fft_buf, fft_buf + nf * nl * S, nf * nl, S, 1, twv + K.tw_y);
    auto neg = [&](int k) { return k == 0 ? 0 : S - k; };
    for (int i = threadIdx.x; i < nl * S; i += FFT_THREADS) {
        const int t = i / nl, l = i - t * nl, g = it.y + l;
        const int kx = g % hx, ky = dims == 3 ? g / hx : t, kz = dims == 3 ? t : 0;
        const int64_t at = K.site_offset + kx + int64_t(S) * (ky + int64_t(S) * kz);
        const bool both = kx > 0 && 2 * kx < S;
        const int64_t at2 = K.site_offset + neg(kx) + int64_t(S) * (neg(ky) + int64_t(S) * neg(kz));
        const double2 p = Z[l * S + t];
        const double c = (p.x * p.x + p.y * p.y) * K.inv_n;
        acc[at] += c;
        if (both) acc[at2] += c;
        if (nf == 1) continue;
        const double2 X = Z[(nl + l) * S + t], Y = Z[(2 * nl + l) * S + t];
        const double2 W = dims == 3 ? Z[(3 * nl + l) * S + t] : make_double2(0.0, 0.0);
        ModeSpectra m = mode_spectra(wrapk(kx, S), wrapk(ky, S), dims == 3 ? wrapk(kz, S) : 0, X, Y, W, dims, K.inv_n);
        jacc[at] += m.x;
        jacc[jstride + at] += m.lon;
        jacc[2 * jstride + at] += m.tra;
        if (both) {
            if (2 * ky == S || (dims == 3 && 2 * kz == S))
                m = mode_spectra(-kx, wrapk(neg(ky), S), dims == 3 ? wrapk(neg(kz), S) : 0, X, Y, W, dims, K.inv_n);
            jacc[at2] += m.x;
            jacc[jstride + at2] += m.lon;
            jacc[2 * jstride + at2] += m.tra;
        }
    }
}

// Momentum spectra of one sample (Eq. 69 diagnostics): from the transforms
// J_a(k) (complex, one field per component) accumulate per k
//   acc[0][k] += |J_x|^2 / N
//   acc[1][k] += |khat . J|^2 / N                       (0 at k = 0)
//   acc[2][k] += (|J|^2 - |khat . J|^2) / (N (d - 1))    (0 at k = 0)
// with khat = n / |n|, n the wrapped integer wavevector; acc[c] = acc + c * stride.
__global__ void __launch_bounds__(AUX_THREADS)
    jk_accum_kernel(const SkSys* __restrict__ skv, const int4* __restrict__ items, int dims,
                    const double* __restrict__ F0, const double* __restrict__ F1, const double* __restrict__ F2,
                    double* __restrict__ acc, int64_t stride) {
    const int4 it = items[blockIdx.x];
    const SkSys K = skv[it.x];
    for (int j = 0; j < SITES_PER_THREAD; ++j) {
        const int e = it.y + j * AUX_THREADS + threadIdx.x;
        if (e >= it.z) break;
        const int64_t g = K.site_offset + e;
        const int kx = e % K.nx, ky = (e / K.nx) % K.ny, kz = e / (K.nx * K.ny);
        const double2 X = make_double2(F0[2 * g], F0[2 * g + 1]), Y = make_double2(F1[2 * g], F1[2 * g + 1]);
        const double2 Z = dims == 3 ? make_double2(F2[2 * g], F2[2 * g + 1]) : make_double2(0.0, 0.0);
        const ModeSpectra m = mode_spectra(wrapk(kx, K.nx), wrapk(ky, K.ny), dims == 3 ? wrapk(kz, K.nz) : 0, X, Y, Z,
                                           dims, K.inv_n);
        acc[g] += m.x;
        acc[stride + g] += m.lon;
        acc[2 * stride + g] += m.tra;
    }
}

// Laplacian of the density deviation d (FP64): lap(r) = 6 sum_i t_i (d(r + c_i) - d(r)).
template <class L>
__global__ void __launch_bounds__(AUX_THREADS)
    jk_lap_kernel(const SysDev* __restrict__ sysv, const int4* __restrict__ items, const double* __restrict__ d,
                  double* __restrict__ lap) {
    const int4 it = items[blockIdx.x];
    const SysDev& S = sysv[it.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz;
    const double* ds = d + S.site_offset;
    for (int j = 0; j < SITES_PER_THREAD; ++j) {
        const int site = it.y + j * AUX_THREADS + threadIdx.x;
        if (site >= it.z) break;
        int x, y, z;
        site_coords(site, nx, ny, x, y, z);
        const double c0 = ds[site];
        double v = 0.0;
#pragma unroll
        for (int i = 1; i < L::Q; ++i) {
            const int sx = wrap1(x + L::c(i, 0), nx), sy = wrap1(y + L::c(i, 1), ny);
            const int sz = L::D == 3 ? wrap1(z + L::c(i, 2), nz) : 0;
            v += 6.0 * L::w(i) * (ds[sx + nx * (sy + ny * sz)] - c0);
        }
        lap[S.site_offset + site] = v;
    }
}

// Guo half-force: j_a(r) += (1/2) kappa rho(r) d_a lap(r), d_a X = 3 sum_i t_i c_ia X(r + c_i),
// rho = rho_c + d; the three components at j + a * stride.
template <class L>
__global__ void __launch_bounds__(AUX_THREADS)
    jk_force_kernel(const SysDev* __restrict__ sysv, const int4* __restrict__ items, const double* __restrict__ d,
                    const double* __restrict__ lap, double* __restrict__ jf, int64_t stride) {
    const int4 it = items[blockIdx.x];
    const SysDev& S = sysv[it.x];
    const int nx = S.nx, ny = S.ny, nz = S.nz;
    const double* ls = lap + S.site_offset;
    for (int j = 0; j < SITES_PER_THREAD; ++j) {
        const int site = it.y + j * AUX_THREADS + threadIdx.x;
        if (site >= it.z) break;
        int x, y, z;
        site_coords(site, nx, ny, x, y, z);
        double g[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int i = 1; i < L::Q; ++i) {
            const int sx = wrap1(x + L::c(i, 0), nx), sy = wrap1(y + L::c(i, 1), ny);
            const int sz = L::D == 3 ? wrap1(z + L::c(i, 2), nz) : 0;
            const double v = ls[sx + nx * (sy + ny * sz)];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                if (L::c(i, a) != 0) g[a] += 3.0 * L::w(i) * double(L::c(i, a)) * v;
        }
        const int64_t gi = S.site_offset + site;
        const double half = 0.5 * S.kappa * (S.rho_c + d[gi]);
#pragma unroll
        for (int a = 0; a < L::D; ++a) jf[a * stride + gi] += half * g[a];
    }
}

// Shell sums of one system's accumulated spectra: CTA (j - 1, c) adds the
// points of shell j, j (j - 1) < |n|^2 <= j (j + 1), of spectrum c (at acc + c
// stride) in a fixed order, one row (ky, kz) per thread at a time: the row's
// points of the shell are the two runs kx = +-(a .. b).  (Every CTA tested
// every k point before: 0.5 ms for 32 shells of 64^3.)
__global__ void __launch_bounds__(AUX_THREADS)
    sk_bin_kernel(const SkSys* __restrict__ skv, int sys, const double* __restrict__ acc, int64_t stride,
                  double* __restrict__ sums, double* __restrict__ counts) {
    __shared__ BlockSum<2, AUX_THREADS> sh;
    const SkSys K = skv[sys];
    const int64_t j = blockIdx.x + 1, lo = j * (j - 1), hi = j * (j + 1);
    const int S = K.nx;
    const double* row0 = acc + blockIdx.y * stride + K.site_offset;
    double v[2] = {0.0, 0.0};
    for (int r = threadIdx.x; r < K.ny * K.nz; r += AUX_THREADS) {
        const int64_t ny = wrapk(r % K.ny, K.ny), nz = wrapk(r / K.ny, K.nz), m = ny * ny + nz * nz;
        if (m > hi) continue;
        // smallest and largest x >= 0 with lo < x^2 + m <= hi
        int b = int(sqrt(double(hi - m)));
        while (int64_t(b) * b > hi - m) --b;
        while (int64_t(b + 1) * (b + 1) <= hi - m) ++b;
        int a = 0;
        if (m <= lo) {
            a = int(sqrt(double(lo - m)));
            while (int64_t(a) * a > lo - m) --a;
            while (int64_t(a) * a + m <= lo) ++a;
        }
        const double* row = row0 + int64_t(S) * r;
        for (int x = a; x <= b && 2 * x <= S; ++x) {
            if (2 * x < S) {                              // wrapped components -S/2 .. (S - 1)/2
                v[0] += row[x];
                v[1] += 1.0;
            }
            if (x > 0) {
                v[0] += row[S - x];
                v[1] += 1.0;
            }
        }
    }
    block_sum(v, sh);
    if (threadIdx.x == 0) {
        sums[blockIdx.y * gridDim.x + blockIdx.x] = v[0];
        counts[blockIdx.y * gridDim.x + blockIdx.x] = v[1];
    }
}

}  // namespace

cudaError_t launch_sk_twiddles(double* tw, const int* sides, const int* offs, int n_tables, int max_n,
                               cudaStream_t st) {
    if (n_tables == 0) return cudaSuccess;
    dim3 grid((max_n + 255) / 256, n_tables);
    sk_twiddle_kernel<<<grid, 256, 0, st>>>(tw, sides, offs, n_tables, max_n);
    return cudaGetLastError();
}

cudaError_t launch_sk_x(const SkSys* sk, const int4* items, int n_items, const double* d,
                        const double* dbar, const double* tw, double* out, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    sk_x_kernel<<<n_items, AUX_THREADS, 0, st>>>(sk, items, d, dbar, tw, out);
    return cudaGetLastError();
}

cudaError_t launch_sk_pass(const SkSys* sk, const int4* items, int n_items, int axis, const double* tw,
                           const double* in, double* out, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    sk_pass_kernel<<<n_items, AUX_THREADS, 0, st>>>(sk, items, axis, tw, in, out);
    return cudaGetLastError();
}

bool sk_fft_side(int n) { return n >= 1 && n <= kSkFftMaxElems; }

cudaError_t launch_sk_fft(const FftLaunch& a, cudaStream_t st) {
    // two buffers of kSkFftMaxElems values; the last pass holds every field of a
    // line, three of kSkFftMaxElems in 2-D (192 KB), four of at most 483 in 3-D
    constexpr int kMaxBytes = int(2 * kSkFftMaxElems * sizeof(double2));
    static PerDevice attr;
    cudaError_t e = cudaSuccess;
    const int set = attr.get(current_device(), [&] {
        e = cudaFuncSetAttribute(fft_x_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxBytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fft_y_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxBytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fft_last_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 3 * kMaxBytes);
        return e == cudaSuccess ? 1 : 0;
    });
    if (!set) return e;
    const double2* tw = reinterpret_cast<const double2*>(a.tw);
    double2* F = reinterpret_cast<double2*>(a.F);
    // both line buffers of the largest item
    const size_t line = 2 * sizeof(double2);
    fft_x_kernel<<<a.n_x, FFT_THREADS, line * a.max_x, st>>>(a.sk, a.items, a.d, a.dbar, a.j, a.n_sites, tw, F,
                                                            a.fstride);
    e = cudaGetLastError();
    if (e == cudaSuccess && a.dims == 3) {
        fft_y_kernel<<<a.n_y, FFT_THREADS, line * a.max_y, st>>>(a.sk, a.items + a.n_x, tw, F, a.fstride);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    fft_last_kernel<<<a.n_last, FFT_THREADS, line * a.max_last, st>>>(a.sk, a.items + a.n_x + a.n_y, a.nf, tw, F,
                                                                      a.fstride, a.acc, a.jacc, a.n_sites, a.dims);
    return cudaGetLastError();
}

cudaError_t launch_sk_accum(const SkSys* sk, const int4* items, int n_items, const double* F, double* acc,
                            cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    sk_accum_kernel<<<n_items, AUX_THREADS, 0, st>>>(sk, items, F, acc);
    return cudaGetLastError();
}

cudaError_t launch_jk_accum(const SkSys* sk, const int4* items, int n_items, int dims, const double* F0,
                            const double* F1, const double* F2, double* acc, int64_t stride, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    jk_accum_kernel<<<n_items, AUX_THREADS, 0, st>>>(sk, items, dims, F0, F1, F2, acc, stride);
    return cudaGetLastError();
}

cudaError_t launch_jk_guo_force(int lattice, const SysDev* sys, const int4* items, int n_items, const double* d,
                                double* lap, double* jf, int64_t stride, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    if (lattice == 0) {
        jk_lap_kernel<D2Q9><<<n_items, AUX_THREADS, 0, st>>>(sys, items, d, lap);
        jk_force_kernel<D2Q9><<<n_items, AUX_THREADS, 0, st>>>(sys, items, d, lap, jf, stride);
    } else {
        jk_lap_kernel<D3Q19><<<n_items, AUX_THREADS, 0, st>>>(sys, items, d, lap);
        jk_force_kernel<D3Q19><<<n_items, AUX_THREADS, 0, st>>>(sys, items, d, lap, jf, stride);
    }
    return cudaGetLastError();
}

cudaError_t launch_sk_bin(const SkSys* sk, int sys, const double* acc, int64_t stride, int nspec, int nbins,
                          double* sums, double* counts, cudaStream_t st) {
    if (nbins <= 0) return cudaSuccess;
    sk_bin_kernel<<<dim3(nbins, nspec), AUX_THREADS, 0, st>>>(sk, sys, acc, stride, sums, counts);
    return cudaGetLastError();
}

}  // namespace lbf

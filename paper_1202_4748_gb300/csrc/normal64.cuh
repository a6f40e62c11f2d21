// Standard normals of the FP64 path in 64-bit integer arithmetic.
//
// Box-Muller of two 32-bit words, R = sqrt(-2 ln U_a), n = R (cos, sin)(2 pi U_b)
// with U = (w + 1/2) 2^-32.  GB300's FP64 units do two operations per clock and
// SM against 128 or more of its integer ones, and the library logarithm, square
// root, sine and cosine of a pair are about 70 FP64 operations, 560 of the 930
// per site of a D3Q19 step.  The words are integers, so everything up to the
// final products is done in fixed point here: four FP64 operations per pair
// with the scale, the rest on the integer units beside them.
//
// Methods (all from the series' definitions):
//  * logarithm: U = f 2^-p, f in [1/2, 1); with c = C/256 from a table on f's six
//    leading bits such that f c <= 1, z = 1 - f c is exact (41 bits) and
//    -ln U = p ln 2 + ln c + z + z^2/2 + z^3/3 + ...: every term is positive and
//    near U = 1 (c = 1, p = 0) the sum is z (1 + z/2 + ...) with exact z, so the
//    result keeps its relative accuracy; terms to z^10/10 with z < 0.018;
//  * square root: a 22-bit reciprocal square root y of the mantissa from the
//    special-function unit, then sqrt(v) = v y (1 - e)^(-1/2), e = 1 - v y^2,
//    with the e and e^2 terms (e^3 is below 2^-62);
//  * sine and cosine: the angle's octant by its top bits, then the Taylor series
//    in w = t^2 of the angle (pi/4) t, t in (0, 1) an exact 30-bit fraction; the
//    sine as t S(w), so small sines keep their relative accuracy.
// R, cos and sin are formed to about 2^-58 and rounded once to double, which is
// closer to the exact values than the library functions' chain (their errors
// are 1 to 2 units in the last place each).
#pragma once

#include <cstdint>
#include <cstring>
#include <type_traits>

#ifdef __CUDACC__
#define LB_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#define LB_HD inline
#endif

namespace lbf {

struct LogEntry {
    uint32_t C;         // floor(2^15 / (65 + i)): c = C / 256 <= 1 / f on f in [(64 + i)/128, (65 + i)/128)
    uint64_t lnc;       // ln(c) 2^64
};

// (a * b) >> 64, (a * b) >> 32
LB_HD uint64_t n64_mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return uint64_t((unsigned __int128)(a) * b >> 64);
#endif
}
LB_HD int64_t n64_smulhi(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return int64_t((__int128)(a) * b >> 64);
#endif
}
LB_HD uint32_t n64_mulhi32(uint32_t a, uint32_t b) { return uint32_t(uint64_t(a) * b >> 32); }
LB_HD int n64_clz(uint64_t a) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)a);
#else
    return __builtin_clzll(a);
#endif
}
LB_HD double n64_bits(uint64_t u) {
    double d;
    memcpy(&d, &u, 8);
    return d;
}
LB_HD float n64_rsqrt(float x) {
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / std::sqrt(x);
#endif
}

// (m / 2^64) 2^e rounded to double, m in [2^63, 2^64) (2^63 - 4 and above round to it)
LB_HD double n64_double(uint64_t m, int e) {
    return n64_bits((uint64_t(e + 1021) << 52) + (m >> 11) + ((m >> 10) & 1));
}

// y (1 - e)^(-1/2) - y in Q62 terms: for v in [1/4, 1) (Q64) the seed y (Q23,
// about 22 bits) and c = (1 - e)^(-1/2) - 1 in Q61, e = 1 - v y^2
LB_HD void n64_seed(uint64_t v, uint32_t& y, int64_t& c) {
    y = uint32_t(n64_rsqrt(float(uint32_t(v >> 40)) * 5.9604644775390625e-08f) * 8388608.0f);
    const int64_t e = int64_t((uint64_t(1) << 61) - n64_mulhi(v, (uint64_t(y) * y) << 15));                    // Q61
    const int64_t eh = e >> 10;
    c = (e >> 1) + ((3 * ((eh * eh) >> 41)) >> 3);
}

// sqrt(v / 2^64) as Q64, v in [2^62, 2^64)
LB_HD uint64_t n64_root(uint64_t v) {
    uint32_t y;
    int64_t c;
    n64_seed(v, y, c);
    const uint64_t r0 = n64_mulhi(v, uint64_t(y) << 39);                                                       // Q62
    uint64_t r = r0 + uint64_t(n64_smulhi(int64_t(r0), c * 8));
    const uint64_t top = (uint64_t(1) << 62) - 1;
    r = r > top ? top : r;
    return r << 2;
}

// sqrt(x) of a positive normal x, correctly rounded, and 1/sqrt(x), within 0.51
// units in the last place (16 and 10 FP64 operations of the library become integer
// ones); anything else through the library.
LB_HD bool n64_split(double x, uint64_t& v, int& h) {
    uint64_t u;
    memcpy(&u, &x, 8);
    const uint32_t eb = uint32_t(u >> 52);
    if (eb - 1u >= 0x7feu) return false;                       // zero, subnormal, negative, infinite or NaN
    // x = (m / 2^64) 2^(eb - 1022) = v 2^(2h)
    const uint64_t m = (u | (uint64_t(1) << 52)) << 11;
    const int e = int(eb) - 1022;
    v = (e & 1) ? m >> 1 : m;
    h = (e + 1) >> 1;
    return true;
}
LB_HD double n64_sqrt(double x) {
    uint64_t v;
    int h;
    if (!n64_split(x, v, h)) return sqrt(x);
    // the nearest 53-bit N of the root to 2^-58, then of the exact one: the root
    // lies below N + 1/2 (N - 1/2) where v 2^44 does below (2N + 1)^2 ((2N - 1)^2),
    // all modulo 2^64 (the differences are below 2^57; no root of 53 bits is a half)
    const uint64_t r = n64_root(v);
    uint64_t N = (r >> 11) + ((r >> 10) & 1);
    const int64_t d = int64_t((v << 44) - 4 * N * N);
    N += uint64_t(d > int64_t(4 * N)) - uint64_t(d < -int64_t(4 * N));
    return n64_bits((uint64_t(h + 1021) << 52) + N);
}
LB_HD double n64_inv_sqrt(double x) {
    uint64_t v;
    int h;
    if (!n64_split(x, v, h)) return 1.0 / sqrt(x);
    uint32_t y;
    int64_t c;
    n64_seed(v, y, c);
    const uint64_t y62 = uint64_t(y) << 38;                    // y / 2 (y in (1, 2]) as Q62
    uint64_t r = y62 + uint64_t(n64_smulhi(int64_t(y62), c * 8));
    const uint64_t top = (uint64_t(1) << 62) - 1;
    r = r > top ? top : r;
    return n64_double(r << 2, 1 - h);
}

// Sums of N floats or doubles to about 2^-57 of the largest: the mantissas
// aligned to the largest exponent as integers of 58 bits, so that a sum of up to
// 31 of them fits 63 bits and every sum costs integer additions (floats within
// 2^-34 of the largest enter exactly).  Subnormal values count as 0 and a sum has
// to be a normal double, which holds in_range(): where the largest value is so
// small that subnormal ones matter beside it, so large that a sum may overflow,
// infinite or NaN (finite() is false), the sums are the caller's in FP64.
template <class T, int N>
struct FixedSum {
    static_assert(N <= 31, "headroom");
    using Bits = typename std::conditional<sizeof(T) == 8, uint64_t, uint32_t>::type;
    static constexpr int kMant = sizeof(T) == 8 ? 52 : 23;            // stored mantissa bits
    static constexpr int kExp = sizeof(T) == 8 ? 20 : 23;             // exponent's place in the high word
    static constexpr uint32_t kTop = sizeof(T) == 8 ? 0x7ff00000u : 0x7f800000u;
    static constexpr int kBias = sizeof(T) == 8 ? 1023 : 127;
    int64_t m[N];
    uint32_t top;                  // largest exponent field, in place
    static LB_HD uint32_t high(Bits u) {
        if constexpr (sizeof(T) == 8) return uint32_t(u >> 32);
        else return u;
    }
    LB_HD explicit FixedSum(const T (&f)[N]) {
        Bits u[N];
        top = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int i = 0; i < N; ++i) {
            memcpy(&u[i], &f[i], sizeof(T));
            const uint32_t e = high(u[i]) & kTop;
            top = e > top ? e : top;
        }
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int i = 0; i < N; ++i) {
            const uint32_t hi = high(u[i]), e = hi & kTop;
            const uint32_t sh = (top - e) >> kExp;
            // zeros and subnormals count as 0
            const Bits one = Bits(1) << kMant;
            const uint64_t a = e ? uint64_t((u[i] & (one - 1)) | one) << (57 - kMant) : 0;
            const uint64_t half = (uint64_t(1) << (sh & 63)) >> 1;
            const int64_t v = sh > 58 ? 0 : int64_t((a + half) >> (sh & 63));
            m[i] = int32_t(hi) < 0 ? -v : v;
        }
    }
    LB_HD bool finite() const { return top != kTop; }
    // largest value from 2^63 times the subnormal ones (doubles: and its 2^-57 a normal double) to 2^-5 of overflow
    LB_HD bool in_range() const {
        constexpr uint32_t low = 64u << kExp, high = sizeof(T) == 8 ? 2040u << kExp : kTop;
        return top - low < high - low;
    }
    // the double nearest to s 2^(top - bias - 57)
    LB_HD double value(int64_t s) const {
        if (s == 0) return 0.0;
        const uint64_t a = s < 0 ? uint64_t(0) - uint64_t(s) : uint64_t(s);
        const int nl = n64_clz(a), e = int(top >> kExp) - kBias + 1 - 57 + 63 - nl;      // (m / 2^64) 2^e
        const double d = n64_double(a << nl, e);
        return s < 0 ? -d : d;
    }
};

// Sums of N doubles to about 2^-116 of the largest, rounded once (to nearest,
// ties to even): as FixedSum with 122 bits, for sums whose cancellation has to
// keep its digits (a site's momentum is often far below its populations).  The
// integers are formed one by one, add(i) at a time, so that a site needs no array
// of them.  (Compensated FP64 sums, to 2^-106, cost six FP64 operations an addend.)
template <int N>
struct WideSum {
    static_assert(N <= 31, "headroom");
    const double (&f)[N];
    uint32_t top;                  // largest exponent field, in place
    static LB_HD uint64_t bits(double x) {
        uint64_t u;
        memcpy(&u, &x, 8);
        return u;
    }
    LB_HD explicit WideSum(const double (&v)[N]) : f(v), top(0) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int i = 0; i < N; ++i) {
            const uint32_t e = uint32_t(bits(f[i]) >> 32) & 0x7ff00000u;
            top = e > top ? e : top;
        }
    }
    LB_HD bool finite() const { return top != 0x7ff00000u; }
    // as FixedSum: 2^-121 of the largest value is a normal double, 2^5 times it too
    LB_HD bool in_range() const {
        constexpr uint32_t low = 160u << 20, high = 2040u << 20;
        return top - low < high - low;
    }
    // f[i] as an integer multiple of 2^(top - bias - 121)
    LB_HD __int128 add(int i) const {
        const uint64_t u = bits(f[i]), one = uint64_t(1) << 52;
        const uint32_t e = uint32_t(u >> 32) & 0x7ff00000u, sh = (top - e) >> 20;
        if (e == 0 || sh > 121) return 0;                  // zeros and subnormals count as 0
        const __int128 v = __int128((unsigned __int128)((u & (one - 1)) | one) << 69 >> sh);
        return int64_t(u) < 0 ? -v : v;
    }
    LB_HD double value(__int128 s) const {
        if (s == 0) return 0.0;
        unsigned __int128 a = s < 0 ? -(unsigned __int128)s : (unsigned __int128)s;
        const int nl = uint64_t(a >> 64) ? n64_clz(uint64_t(a >> 64)) : 64 + n64_clz(uint64_t(a));
        a <<= nl;
        const uint64_t m = uint64_t(a >> 64), rest = (m & 0x3ff) | (uint64_t(a) != 0) | ((m >> 11) & 1);
        const int e = int(top >> 20) - 1023 + 1 - 121 + 127 - nl;                          // (m / 2^64) 2^e
        const double d = n64_bits((uint64_t(e + 1021) << 52) + (m >> 11) + (((m >> 10) & 1) & (rest != 0)));
        return s < 0 ? -d : d;
    }
};

// sqrt(-2 ln U), U = (w + 1/2) 2^-32; tab holds the 64 entries of kLogTable
template <class Table>
LB_HD double n64_radius(uint32_t w, const Table& tab) {
    // U = (Y / 2^64) 2^-p, Y in [2^63, 2^64) with its 33 leading bits significant
    const uint64_t M = 2 * uint64_t(w) + 1;
    const int k = n64_clz(M), p = k - 31;
    const uint64_t Y = M << k;
    const LogEntry t = tab(int(Y >> 57) & 63);
    const uint64_t z = ((uint64_t(1) << 41) - (Y >> 31) * t.C) << 23;              // Q64
    // P = 1/2 + z/3 + ... + z^8/10
    const uint32_t z32 = uint32_t(z >> 32);
    uint32_t a = 429496730u;                                                        // 1/10
    a = 477218588u + n64_mulhi32(z32, a);                                           // 1/9
    a = 536870912u + n64_mulhi32(z32, a);                                           // 1/8
    a = 613566757u + n64_mulhi32(z32, a);                                           // 1/7
    a = 715827883u + n64_mulhi32(z32, a);                                           // 1/6
    uint64_t P = 0x3333333333333333ull + n64_mulhi(z, uint64_t(a) << 32);           // 1/5
    P = 0x4000000000000000ull + n64_mulhi(z, P);                                    // 1/4
    P = 0x5555555555555555ull + n64_mulhi(z, P);                                    // 1/3
    P = 0x8000000000000000ull + n64_mulhi(z, P);                                    // 1/2
    const uint64_t zP = n64_mulhi(z, P);
    // -ln U = L 2^-q: q = 59 for U < 1/2, 63 below f = 127/128, else as many as z allows
    const bool one = p == 0 && t.C == 256;
    const int s = p == 0 ? 1 : 5, cz = n64_clz(z | 1) - 1;
    const uint64_t zt = one ? z << cz : z >> s;
    const int q = one ? 64 + cz : 64 - s;
    const uint64_t base = uint64_t(p) * 0x058b90bfbe8e7bcdull + (t.lnc >> s);
    uint64_t L = base + zt + n64_mulhi(zt, zP);
    const int nl = n64_clz(L);
    L <<= nl;
    // 2 (-ln U) = v 2^(2h), v in [1/4, 1) as Q64
    const int g = 65 - q - nl, h = (g + 1) >> 1;
    return n64_double(n64_root((g & 1) ? L >> 1 : L), h);
}

// cos and sin of 2 pi U, U = (w + 1/2) 2^-32
LB_HD void n64_angle(uint32_t w, double& co, double& si) {
    const uint32_t o = w >> 29;
    uint32_t T = (2u * w + 1u) & 0x3fffffffu;                 // position in the octant, odd
    if (o & 1) T = 0x40000000u - T;                           // t = T / 2^30
    const uint64_t W = (uint64_t(T) * T) << 4;                // t^2, Q64
    const uint32_t W32 = uint32_t(W >> 32);
    uint32_t a = 53u;                                        // (pi/4)^(2k+1)/(2k+1)!, k = 8 .. 5, Q60
    a = 23531u - n64_mulhi32(W32, a);
    a = 8011021u - n64_mulhi32(W32, a);
    a = 2025968632u - n64_mulhi32(W32, a);
    uint64_t S = 0x00000541e0d21fbaull - n64_mulhi(W, uint64_t(a) << 4);       // k = 4 .. 0, Q64
    S = 0x000265a599cc57b1ull - n64_mulhi(W, S);
    S = 0x00a335e33bad570full - n64_mulhi(W, S);
    S = 0x14abbce625be52bfull - n64_mulhi(W, S);
    S = 0xc90fdaa22168c235ull - n64_mulhi(W, S);
    uint32_t b = 2u;                                        // (pi/4)^(2k)/(2k)!, k = 9 .. 6, Q60
    b = 1155u - n64_mulhi32(W32, b);
    b = 449417u - n64_mulhi32(W32, b);
    b = 132599337u - n64_mulhi32(W32, b);
    uint64_t C = 0x00000069b47ca881ull - n64_mulhi(W, uint64_t(b) << 4);       // k = 5 .. 1, Q64
    C = 0x00003c3ea0d12375ull - n64_mulhi(W, C);
    C = 0x00155d3c7e3cbffaull - n64_mulhi(W, C);
    C = 0x040f07c206d6b0edull - n64_mulhi(W, C);
    C = 0x4ef4f326f9177969ull - n64_mulhi(W, C);
    C = 0ull - n64_mulhi(W, C);                               // cos in (0.7, 1), Q64 (t > 0: below 1)
    // sin = t S, normalised
    const int cz = n64_clz(T) - 32;
    uint64_t m = n64_mulhi(S, uint64_t(T) << (32 + cz));
    const int nl = n64_clz(m);
    const double c = n64_double(C, 0), s = n64_double(m << nl, 2 - cz - nl);
    const bool swap = ((o + 1) >> 1) & 1;
    const double x = swap ? s : c, y = swap ? c : s;
    co = ((o + 2) >> 2) & 1 ? -x : x;
    si = o >> 2 ? -y : y;
}

#define LB_LOG_TABLE \
    {504u, 0xad6a0261acf967d9ull}, {496u, 0xa9516932de2d5774ull}, {489u, 0xa5adeb4ab7139c6full}, \
    {481u, 0xa174e36efc05f965ull}, {474u, 0x9db4224fffe1157cull}, {468u, 0x9a7144ece70e98b7ull}, \
    {461u, 0x9695a00976e4ed5eull}, {455u, 0x933b1009a186fe69ull}, {448u, 0x8f42faf3820681efull}, \
    {442u, 0x8bcf55dec4cd05feull}, {436u, 0x884f9cf16a64b7efull}, {431u, 0x855bb5f670a68e03ull}, \
    {425u, 0x81c4f77e7319d9e1ull}, {420u, 0x7ebd623de3cc7b67ull}, {414u, 0x7b0e67491a33005dull}, \
    {409u, 0x77f216641b56d502ull}, {404u, 0x74cbf9f803af5587ull}, {399u, 0x719bd38ffdbfdf9full}, \
    {394u, 0x6e61625a4c43ed66ull}, {390u, 0x6bc4a4c91de1ac45ull}, {385u, 0x6877019356e65590ull}, \
    {381u, 0x65ca8d044d4561a6ull}, {376u, 0x6268ce1b05096ad7ull}, {372u, 0x5fabe0ee0abf0d93ull}, \
    {368u, 0x5ce75fdaef401a74ull}, {364u, 0x5a1b207a6c52bb11ull}, {360u, 0x5746f6fd60272942ull}, \
    {356u, 0x546ab61cb7e0b427ull}, {352u, 0x51862f08717b09f4ull}, {348u, 0x4e993155a517a71dull}, \
    {344u, 0x4ba38aeb8474c271ull}, {341u, 0x496580437dd8e7bcull}, {337u, 0x466034b7508dbd9dull}, \
    {334u, 0x44162fe6b92b5462ull}, {330u, 0x41009652d341036cull}, {327u, 0x3eaa14ac96f66e0eull}, \
    {324u, 0x3c4e0edc55e5cbd4ull}, {321u, 0x39ec6a9c138bb892ull}, {318u, 0x37850ce85b19ac54ull}, \
    {315u, 0x3517d9f9105e3186ull}, {312u, 0x32a4b539e8ad68edull}, {309u, 0x302b814286afd5adull}, \
    {306u, 0x2dac1fce33a4391bull}, {303u, 0x2b2671b330410ba7ull}, {300u, 0x289a56d996fa3cd0ull}, \
    {297u, 0x2607ae31c8ffa5fdull}, {295u, 0x244cde3214b596fbull}, {292u, 0x21aefcf9a11cb2cdull}, \
    {289u, 0x1f0a30c01162a661ull}, {287u, 0x1d4313d66cb35d5eull}, {284u, 0x1a926d3a4ad56365ull}, \
    {282u, 0x18c345d6319b20f6ull}, {280u, 0x16f0d28ae56b4b9cull}, {277u, 0x142edcbea646f03cull}, \
    {275u, 0x1253f62f0a1416f9ull}, {273u, 0x1075983598e47130ull}, {270u, 0x0da16eb88cb8df61ull}, \
    {268u, 0x0bba2c7b196e7e23ull}, {266u, 0x09cf43dcff5eafd5ull}, {264u, 0x07e0a6c39e0cc013ull}, \
    {262u, 0x05ee46c1f56c46aaull}, {260u, 0x03f815161f807c7aull}, {258u, 0x01fe02a6b1067890ull}, \
    {256u, 0x0000000000000000ull},

}  // namespace lbf

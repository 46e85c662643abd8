// gbpf_fx.cuh -- fixed-point arithmetic of the nodal power-flow quantities.
//
// On GB300 an FP64 instruction of any kind -- multiply-add, conversion,
// compare -- holds its SM sub-partition for 64 cycles, a 32 x 32 -> 64-bit
// integer multiply-add (IMAD.WIDE) for 2 (both measured, one to eight warps
// per sub-partition).  Voltages are bounded and a row of the admittance
// matrix has a known absolute sum, so sums of their products need no
// floating exponent: 59-bit integers hold them with less rounding error than
// FP64 and a product costs three multiply-adds, 6 cycles.
//
// A number v in units 2^-q is an int64; its limbs are v = h 2^30 + l with l
// in [-2^29, 2^29).  Products keep hh and the two cross terms hl + lh; l l
// (below a quarter of the last kept place) is dropped.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define GBPF_FX __host__ __device__ __forceinline__
#else
#define GBPF_FX inline
#endif

namespace gbpf {

constexpr int kFxV = 58;             // voltages e, f: units 2^-58, |V| < 2
constexpr int kFxRow = 58;           // a row's absolute sum is at most 2^58 units
constexpr double kFxVmax = 1.9375;   // |V| taken are below this (2 less room for rounding)
constexpr int kFxNoScale = 4000;     // the scale of a row that has none (not finite, or beyond 2^+-400)
constexpr double kFxThMax = 7.75;    // |theta| of fx_sincos are below this

GBPF_FX unsigned long long fx_umulhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return static_cast<unsigned long long>((static_cast<unsigned __int128>(a) * b) >> 64);
#endif
}
GBPF_FX int fx_clz(unsigned long long a) {
#ifdef __CUDA_ARCH__
    return __clzll(static_cast<long long>(a));
#else
    return a ? __builtin_clzll(a) : 64;
#endif
}
GBPF_FX long long fx_bits(double x) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(x);
#else
    long long b;
    std::memcpy(&b, &x, 8);
    return b;
#endif
}
GBPF_FX double fx_double(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double x;
    std::memcpy(&x, &b, 8);
    return x;
#endif
}

// x in units 2^-q, rounded to nearest (ties away); |x| 2^q < 2^62 and x
// normal, or zero.  Integer instructions only.
GBPF_FX long long fx_from_double(double x, int q) {
    const long long b = fx_bits(x);
    const int ex = int((b >> 52) & 0x7ff);
    const unsigned long long m = (static_cast<unsigned long long>(b) & 0xfffffffffffffull) | (1ull << 52);
    const int sh = ex - 1075 + q;
    unsigned long long a;
    if (sh >= 0) a = m << (sh & 63);
    else a = sh < -54 ? 0ull : ((m >> (-sh - 1)) + 1ull) >> 1;
    if (ex == 0) a = 0ull;
    return b < 0 ? -static_cast<long long>(a) : static_cast<long long>(a);
}
GBPF_FX long long fx_from_double(float x, int q) {
#ifdef __CUDA_ARCH__
    const int b = __float_as_int(x);
#else
    int b;
    std::memcpy(&b, &x, 4);
#endif
    const int ex = (b >> 23) & 0xff;
    const unsigned long long m = (static_cast<unsigned>(b) & 0x7fffffu) | (1u << 23);
    const int sh = ex - 150 + q;
    unsigned long long a;
    if (sh >= 0) a = m << (sh & 63);
    else a = sh < -25 ? 0ull : ((m >> (-sh - 1)) + 1ull) >> 1;
    if (ex == 0) a = 0ull;
    return b < 0 ? -static_cast<long long>(a) : static_cast<long long>(a);
}

// Whether fx_from_double takes x: |x| 2^q below 2^61 and finite.
GBPF_FX bool fx_fits(double x, int q) {
    return int((fx_bits(x) >> 52) & 0x7ff) - 1023 + q < 61;
}

// The double nearest to v 2^-q (ties to even); |q| at most a few hundred.
GBPF_FX double fx_to_double(long long v, int q) {
    if (v == 0) return 0.0;
    const unsigned long long a = v < 0 ? 0ull - static_cast<unsigned long long>(v) : static_cast<unsigned long long>(v);
    const int lz = fx_clz(a);
    const unsigned long long n = a << lz;  // top bit set
    unsigned long long m = n >> 11;
    const unsigned r = unsigned(n) & 0x7ffu;
    m += (r > 0x400u || (r == 0x400u && (m & 1ull))) ? 1ull : 0ull;
    const long long e = 1023 + 63 - lz - q - 1;  // the mantissa's own leading bit adds one
    return fx_double((v < 0 ? static_cast<long long>(1ull << 63) : 0ll) | ((e << 52) + static_cast<long long>(m)));
}

struct FxLimbs {
    int h, l;
};
GBPF_FX FxLimbs fx_split(long long v) {
    FxLimbs r;
    r.l = int(unsigned(static_cast<unsigned long long>(v)) << 2) >> 2;
    r.h = int((v - r.l) >> 30);
    return r;
}
GBPF_FX long long fx_join(int h, int l) { return (static_cast<long long>(h) << 30) + l; }

// Sum of products of limb pairs: hh in units 2^60, mid in units 2^30 of the
// full product's last place.
struct FxAcc {
    long long hh, mid;
};
GBPF_FX void fx_mac(FxAcc &s, int ah, int al, int bh, int bl) {
#ifdef __CUDA_ARCH__
    // as written below, the compiler multiplies and adds in two steps
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s.hh) : "r"(ah), "r"(bh));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s.mid) : "r"(ah), "r"(bl));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s.mid) : "r"(al), "r"(bh));
    return;
#endif
    s.hh += static_cast<long long>(ah) * bh;
    s.mid += static_cast<long long>(ah) * bl;
    s.mid += static_cast<long long>(al) * bh;
}
GBPF_FX void fx_carry(FxAcc &s) {
    s.hh += s.mid >> 30;
    s.mid &= (1ll << 30) - 1;
}
// The sum in units 2^(60 - K) of the product's last place, rounded.
template <int K>
GBPF_FX long long fx_sum(const FxAcc &s) {
    return (s.hh << K) + ((s.mid + (1ll << (29 - K))) >> (30 - K));
}

// sin and cos of x (|x| < kFxThMax) in units 2^-60, within about two units:
// x in units 2^-60, reduced by the nearest multiple of pi/2 (held to 92
// fractional bits), then the Maclaurin series of both in unsigned 0.64
// arithmetic; the terms from x^13 (sin) and x^12 (cos) on need 32 bits.
GBPF_FX void fx_sincos60(long long t, long long &s_out, long long &c_out) {
    const int th = int(t >> 32);  // units 2^-28
    const int k = int(rintf(float(th) * float(0.63661977236758134 / 268435456.0)));
    constexpr long long kPio2 = 1811004864519280710ll;  // floor(pi/2 2^60)
    constexpr long long kPio2Lo = 2560150609ll;         // its next 32 bits
    const long long r = t - k * kPio2 - ((k * kPio2Lo + (1ll << 31)) >> 32);
    const unsigned long long x64 = static_cast<unsigned long long>(r < 0 ? -r : r) << 4;  // |r| < 0.79, 0.64
    const unsigned long long z = fx_umulhi(x64, x64);
    const unsigned z32 = unsigned(z >> 32);
    auto mul32 = [](unsigned a, unsigned b) {
        return unsigned((static_cast<unsigned long long>(a) * b) >> 32);
    };
    // sin r / r: 1/(2k + 1)! in units 2^-64 (32-bit terms), then 2^-63
    unsigned u = 51862u;                        // 2^64 / 17!
    u = 14106527u - mul32(z32, u);              // 2^64 / 15!
    u = 2962370717u - mul32(z32, u);            // 2^64 / 13!
    unsigned long long p = 231064915947ull - fx_umulhi(z, static_cast<unsigned long long>(u) >> 1);  // 2^63 / 11!
    p = 25417140754119ull - fx_umulhi(z, p);    // 2^63 / 9!
    p = 1830034134296583ull - fx_umulhi(z, p);  // 2^63 / 7!
    p = 76861433640456465ull - fx_umulhi(z, p); // 2^63 / 5!
    p = 1537228672809129301ull - fx_umulhi(z, p);  // 2^63 / 3!
    p = 9223372036854775808ull - fx_umulhi(z, p);
    const long long sr = static_cast<long long>((fx_umulhi(x64, p) + 4ull) >> 3);
    // cos r: 1/(2k)! in units 2^-60 (32-bit terms), then 2^-63
    unsigned w = 180u;                          // 2^60 / 18!
    w = 55104u - mul32(z32, w);                 // 2^60 / 16!
    w = 13224869u - mul32(z32, w);              // 2^60 / 14!
    w = 2406926208u - mul32(z32, w);            // 2^60 / 12!
    unsigned long long q = 2541714075412ull - fx_umulhi(z, static_cast<unsigned long long>(w) << 3);  // 2^63 / 10!
    q = 228754266787073ull - fx_umulhi(z, q);   // 2^63 / 8!
    q = 12810238940076078ull - fx_umulhi(z, q); // 2^63 / 6!
    q = 384307168202282325ull - fx_umulhi(z, q);   // 2^63 / 4!
    q = 4611686018427387904ull - fx_umulhi(z, q);
    q = 9223372036854775808ull - fx_umulhi(z, q);
    const long long cr = static_cast<long long>((q + 4ull) >> 3);
    const long long sg = r < 0 ? -sr : sr;
    const long long sn = k & 1 ? cr : sg, cn = k & 1 ? sg : cr;
    s_out = k & 2 ? -sn : sn;
    c_out = (k + 1) & 2 ? -cn : cn;
}

#ifdef __CUDACC__
// The float nearest to v 2^-q for results in a float's normal range: the 32
// leading bits, the last one standing for all that follow, take one 32-bit
// conversion (a 64-bit one costs as much as an FP64 instruction).
__device__ __forceinline__ float fx_to_float(long long v, int q) {
    const unsigned long long a = v < 0 ? 0ull - static_cast<unsigned long long>(v) : static_cast<unsigned long long>(v);
    const int lz = __clzll(static_cast<long long>(a | 1ull));
    const unsigned long long n = a << lz;
    const unsigned m = unsigned(n >> 32) | (unsigned(n) ? 1u : 0u);
    const float f = __int_as_float(__float_as_int(__uint2float_rn(m)) + ((32 - lz - q) << 23));
    return a ? (v < 0 ? -f : f) : 0.0f;
}
// The limbs of x in units 2^-60, |x| < 2.
__device__ __forceinline__ FxLimbs fx_limbs60(float x) {
    const float y = x * 1073741824.0f, h = rintf(y);
    return FxLimbs{__float2int_rn(h), __float2int_rn((y - h) * 1073741824.0f)};
}
#endif

// 1 / v in units 2^-60 for v in units 2^-58, 0.25 < |v| < 2: the FP32
// reciprocal y (within 2^-22) and y (1 + r + r^2), r = 1 - v y; within a few
// units.
GBPF_FX long long fx_recip(long long v) {
    const FxLimbs a = fx_split(v);
#ifdef __CUDA_ARCH__
    const float yf = __frcp_rn(float(a.h));
#else
    const float yf = 1.0f / float(a.h);
#endif
    const int y = int(yf * 18014398509481984.0f);  // units 2^-26: 2^(26 + 28)
    const long long r = (1ll << 60) - (((static_cast<long long>(a.h) * y) << 6) + ((static_cast<long long>(a.l) * y) >> 24));
    const int rs = int(r >> 10);
    const long long c = r + ((static_cast<long long>(rs) * rs) >> 40);
    const int ch = int(c >> 20), cl = int(c & 0xfffff);
    return (static_cast<long long>(y) << 34) + ((static_cast<long long>(y) * ch) >> 6) +
           ((static_cast<long long>(y) * cl) >> 26);
}

// sin d and 1 - cos d in units 2^-60 for d in units 2^-60, |d| <= 0.2, within
// 2.5 and 1 units.  small: |d| < 2^-10.
GBPF_FX void fx_small_sincos(long long d, bool small, long long &sd, long long &cm) {
    const unsigned long long x = static_cast<unsigned long long>(d < 0 ? -d : d) << 4;  // 0.64
    unsigned long long s, c;
    if (small) {
        // z = x^2 (0.64, below 2^44); s = x - x (z / 6 - z^2 / 120), c = z / 2 - z^2 / 24
        const unsigned xh = unsigned(x >> 27), xl = unsigned(x) & 0x7ffffffu;
        const unsigned long long z =
            (static_cast<unsigned long long>(xh) * xh + ((static_cast<unsigned long long>(xh) * xl) >> 26)) >> 10;
        const unsigned zh = unsigned(z >> 12);                                              // units 2^-52
        const unsigned zz = unsigned((static_cast<unsigned long long>(zh) * zh) >> 40);     // 0.64, below 2^24
        const unsigned long long t = ((static_cast<unsigned long long>(zh) * 715827883u) >> 20) - zz / 120u;
        s = x - ((static_cast<unsigned long long>(unsigned(x >> 24)) * unsigned(t >> 10)) >> 30);
        c = (z >> 1) - zz / 24u;
    } else {
        // terms from x^7 (sin) and x^8 (cos) on in 32 bits: z <= 0.04
        const unsigned long long z = fx_umulhi(x, x);
        const unsigned zh = unsigned(z >> 28);  // units 2^-36
        auto mul = [](unsigned a, unsigned b) {
            return unsigned((static_cast<unsigned long long>(a) * b) >> 32);
        };
        // sin: 1/7! - z/9! + z^2/11! in units 2^-43; then 2^-64
        unsigned u = 220361u;                           // 2^43 / 11!
        u = 24239674u - (mul(zh, u) >> 4);              // 2^43 / 9!
        u = 1745256552u - (mul(zh, u) >> 4);            // 2^43 / 7!
        unsigned long long p = 153722867280912930ull - fx_umulhi(z, static_cast<unsigned long long>(u) << 21);  // 2^64 / 5!
        p = 3074457345618258603ull - fx_umulhi(z, p);   // 2^64 / 3!
        s = x - fx_umulhi(x, fx_umulhi(z, p));
        // cos: 1/8! - z/10! + z^2/12! in units 2^-47; then 2^-64
        unsigned w = 293814u;                           // 2^47 / 12!
        w = 38783479u - (mul(zh, w) >> 4);              // 2^47 / 10!
        w = 3490513104u - (mul(zh, w) >> 4);            // 2^47 / 8!
        unsigned long long q = 25620477880152155ull - fx_umulhi(z, static_cast<unsigned long long>(w) << 17);  // 2^64 / 6!
        q = 768614336404564651ull - fx_umulhi(z, q);    // 2^64 / 4!
        c = (z >> 1) - fx_umulhi(z, fx_umulhi(z, q));
    }
    const long long sr = static_cast<long long>((s + 8ull) >> 4);
    sd = d < 0 ? -sr : sr;
    cm = static_cast<long long>((c + 8ull) >> 4);
}

GBPF_FX void fx_sincos(double x, long long &s_out, long long &c_out) {
    fx_sincos60(fx_from_double(x, 60), s_out, c_out);
}

// e = V cos, f = V sin in units 2^-58, from V in units 2^-58 and cos, sin in
// units 2^-60.
GBPF_FX long long fx_scale_v(long long v, long long c) {
    const FxLimbs a = fx_split(v), b = fx_split(c);
    FxAcc s{0, 0};
    fx_mac(s, a.h, a.l, b.h, b.l);
    return fx_sum<0>(s);
}

}  // namespace gbpf

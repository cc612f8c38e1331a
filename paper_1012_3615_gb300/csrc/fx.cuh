// Fixed-point copies of the FP64 hopping fields and spinors (see dslash_fx.cu
// for the format and its bounds).
#pragma once
#include "common.cuh"

namespace bri {

constexpr int FX_BAD = 1 << 20;     // block exponent of a site out of range: an infinity, a NaN, or FX_WIDE
constexpr int FX_ZERO = -(1 << 20);  // ... of a site that is zero
constexpr int FX_WB = 62, FX_PB = 60;  // fraction bits of links and spinors
constexpr int FX_AB = FX_WB + FX_PB - 64;  // of the row sums
// v 2^sh rounded to an integer (|v| 2^sh < 2^63), by shifts: conversions run on
// the FP64 pipe
BRI_D long long fx_int(double v, int sh) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const int e = (int)(bits >> 52) & 0x7ff;
    const unsigned long long m = (bits & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull);
    const int s = max(e, 1) - 1075 + sh, r = min(-s, 63);
    const long long f = (long long)(s >= 0 ? m << s : (m + ((1ull << r) >> 1)) >> r);
    return (long long)bits < 0 ? -f : f;
}
BRI_D int4 fx_split(double re, double im, int sh) {
    // the low word is never INT_MIN, so that limbs can be negated
    const long long a = fx_int(re, sh), b = fx_int(im, sh);
    int4 v;
    v.y = (int)a;
    v.x = (int)((a - v.y) >> 32);
    v.w = (int)b;
    v.z = (int)((b - v.w) >> 32);
    if (v.y == (int)0x80000000) v.y++;
    if (v.w == (int)0x80000000) v.w++;
    return v;
}
// the same with the low limb as an FP32 number in units of the high one
BRI_D int4 fx_split_f(double re, double im, int sh) {
    const long long a = fx_int(re, sh), b = fx_int(im, sh);
    const int al = (int)a, bl = (int)b;
    return make_int4((int)((a - al) >> 32), __float_as_int((float)al * 0x1p-32f), (int)((b - bl) >> 32),
                     __float_as_int((float)bl * 0x1p-32f));
}
BRI_D unsigned abs_hi(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// f 2^sh, rounded to nearest even, by integer operations
BRI_D double fx_double(long long f, int sh) {
    const unsigned long long u = f < 0 ? 0ull - (unsigned long long)f : (unsigned long long)f;
    if (u == 0) return 0.0;
    const int lz = __clzll((long long)u);
    const unsigned long long m = u << lz;  // leading one at bit 63
    const unsigned long long r = (m + 0x3ffull + ((m >> 11) & 1ull)) >> 11;  // 53 bits; 2^53 when it rounds up
    const bool up = r < (1ull << 52);  // m + ... ran over 2^64
    const unsigned long long q = up ? 1ull << 52 : r;
    const unsigned long long e = (unsigned long long)(1023 + 63 - lz + sh + (up ? 1 : 0) - 1);
    return __longlong_as_double((long long)((e << 52) + q + (f < 0 ? 1ull << 63 : 0ull)));
}
// two signed limbs of an integer (the low one never INT_MIN: limbs can be negated)
BRI_D int2 fx_limbs(long long f) {
    int lo = (int)f;
    const int hi = (int)((f - lo) >> 32);
    if (lo == (int)0x80000000) lo++;
    return make_int2(hi, lo);
}
BRI_D long long fx_join(int hi, int lo) { return (long long)hi * (1ll << 32) + lo; }

// largest |row|^2, |column|^2 of a field matrix, as the high word of a double
// (NaN and infinities come out largest)
BRI_D unsigned norm_hi(const double2 w[9]) {
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        m = max(m, abs_hi(cnorm2(w[3 * i]) + cnorm2(w[3 * i + 1]) + cnorm2(w[3 * i + 2])));
        m = max(m, abs_hi(cnorm2(w[i]) + cnorm2(w[3 + i]) + cnorm2(w[6 + i])));
    }
    return m;
}
constexpr unsigned FX_ONE = 0x3ff00010u;  // 1 + 2^-16: a unitary matrix and its rounding

// limb copies are stored in blocks of 32 sites, [..][Vp/32][entries][32] with Vp
// = V rounded up to 32: the entries of a site lie at fixed offsets from its first
BRI_D size_t fx_at(int site, int entries) { return (size_t)(site >> 5) * (32 * entries) + (site & 31); }

// the limbs of a field matrix of one site (o: the field's start)
BRI_D void fx_store(const double2 w[9], int4 *o, int site) {
    o += fx_at(site, 9);
#pragma unroll
    for (int e = 0; e < 9; e++) o[32 * e] = fx_split_f(w[e].x, w[e].y, FX_WB);
}

}  // namespace bri
